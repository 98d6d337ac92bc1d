// FP64 multipole-to-local over lists of translations sorted by operator.
//
// A translation is one (target box, offset, source type) with charges of that type in the source box.  All
// translations of one operator (class and source type) of a (group, level) job are gathered into
// batches of PAIR_C columns, whatever targets they belong to; one CTA multiplies a batch by the
// operator and writes every column's translated expansion to the translation's own slot.  Slots are
// numbered target by target in (offset, type) order and summed in that order (k_pair_sum), so the
// result does not depend on the order in which the lists were filled.
//
// Bound: the FP64 pipe (0.63 T FMA/s on this GPU, 64 times below FP32), so what counts is the number of
// FMAs issued, not the operand traffic: a batch reads its operator once from L2 (70 KB at p = 10, about 4
// bytes per clock and SM).  Hence no padding to a tile of targets: tiles of 32 targets x 80 rows
// per offset spend most of the pipe on absent sources where boxes hold a few points (2,003 charges at
// p = 12: 252 ms per evaluation for 0.6 M translations of six types, most of them absent).
// Real form: P acts on real parts (K x K) and Q on imaginary parts of the m > 0 coefficients
// (the m = 0 imaginary parts vanish for real charges): K^2 + (K - p - 1)^2 FMAs, not 2 K^2.
#pragma once

// Columns of a batch: two threads per operator row, every other column each, so that a partial batch of n columns
// costs ceil(n / 2) quarters of a full one, not all of it (first and second half each: N = 2,003 p = 12 adjoint 52.5 ms,
// so 49.5; N = 100,000 p = 10 87.7 -> 86.0).
constexpr int PAIR_C = 8;
__device__ __forceinline__ int pair_pos(int c) { return (c & 1) * (PAIR_C / 2) + (c >> 1); }
constexpr uint64_t PAIR_WINDOW_MIN = 4096;  // translations below which a window is not halved for want of memory
constexpr int PAIR_KC = 16;  // operator columns staged at a time (16 doubles = one 128-byte line per row)

struct PairJob {
  const int32_t *vlist;      // [ntb][NOFF] source box or -1
  const int32_t *cls;        // [NOFF] (free) or [NKT][NOFF] (reaction, row ktrow[t]) operator class or -1
  const int32_t *ktrow;      // reaction: target row k_t of every box (nullptr: free)
  const uint32_t *tmask;     // [nsb] source types present (nullptr: type 0 of every box)
  const double2 *M;          // [nsb][ntypes][K]
  const double *ops;         // [ncls][ntypes][2][K][K]
  double2 *L;                // [ntb][K], added to
  int64_t t0;                // first target of this job in the flattened target range
  int32_t ntb, ntypes, nkt, bin0;  // bin0: first bin (class x type) of this job
};

// operator class of (target t, offset o), or -1
__device__ __forceinline__ int pair_class(const PairJob &J, int64_t t, int o) {
  if (!J.ktrow) return J.cls[o];
  const int kt = J.ktrow[t];
  return (kt >= 0 && kt < J.nkt) ? J.cls[(size_t)kt * NOFF + o] : -1;
}
__device__ __forceinline__ int pair_find_job(const PairJob *jobs, int njobs, int64_t g) {
  int lo = 0, hi = njobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].t0 <= g) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// MODE 0: translations of every target (cnt[g]); 1: bin counts of the translations numbered
// [w0, w1); 2: those translations into their bins' lists.  One warp per target.
struct PairEnt {
  uint32_t e;  // slot (relative to the window)
  int32_t s;   // source box
  int32_t o;   // offset
};
template <int MODE>
__global__ void k_pair_walk(const PairJob *jobs, int njobs, int64_t ntot, uint32_t *cnt, const uint32_t *e0,
                            uint32_t w0, uint32_t w1, uint32_t *bins, const uint32_t *bin_batch, PairEnt *list) {
  const int64_t g = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (g >= ntot) return;
  const int lane = threadIdx.x & 31;
  uint32_t e = MODE ? e0[g] : 0u, total = 0;
  if (MODE && (e >= w1 || e + cnt[g] <= w0)) return;  // no translation of this target in the window
  const PairJob &J = jobs[pair_find_job(jobs, njobs, g)];
  const int64_t t = g - J.t0;
  if (!J.ktrow || (J.ktrow[t] >= 0 && J.ktrow[t] < J.nkt)) {
    for (int o0 = 0; o0 < NOFF; o0 += 32) {
      const int o = o0 + lane;
      const int s = o < NOFF ? J.vlist[(size_t)t * NOFF + o] : -1;
      const int cls = s >= 0 ? pair_class(J, t, o) : -1;
      const uint32_t m = cls < 0 ? 0u : (J.tmask ? J.tmask[s] : 1u);
      const uint32_t c = __popc(m);
      if (MODE == 0) {
        total += c;
      } else {
        uint32_t x = c;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
          if (lane >= d) x += y;
        }
        uint32_t my = e + x - c;
        for (uint32_t r = m; r; r &= r - 1, ++my) {
          if (my < w0 || my >= w1) continue;
          const int bin = J.bin0 + cls * J.ntypes + (__ffs(r) - 1);
          const uint32_t pos = atomicAdd(&bins[bin], 1u);
          if (MODE == 2) list[(size_t)bin_batch[bin] * PAIR_C + pos] = PairEnt{my - w0, s, o};
        }
        e += __shfl_sync(0xffffffffu, x, 31);
      }
    }
  }
  if (MODE == 0) {
    total = wsum(total);
    if (lane == 0) cnt[g] = total;
  }
}

__global__ void k_pair_batches(const uint32_t *bins, int nbins, uint32_t *nbatch) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < nbins) nbatch[b] = (bins[b] + PAIR_C - 1) / PAIR_C;
}

// acc[j] += W(row, k) X(k, j) over kn operator columns for the first CN of a thread's columns
template <int CN>
__device__ __forceinline__ void pair_dot(double *acc, const double *w, int ld, const double *x, int kn) {
#pragma unroll 4
  for (int kk = 0; kk < kn; ++kk) {
    const double wv = w[kk * ld];
    const double2 xa = *(const double2 *)(x + kk * PAIR_C);
    acc[0] = fma(wv, xa.x, acc[0]);
    if (CN > 1) acc[1] = fma(wv, xa.y, acc[1]);
    if (CN > 2) {
      const double2 xc = *(const double2 *)(x + kk * PAIR_C + 2);
      acc[2] = fma(wv, xc.x, acc[2]);
      if (CN > 3) acc[3] = fma(wv, xc.y, acc[3]);
    }
  }
}

// One CTA per batch: 2 threads per real operator row, PAIR_C / 2 columns each.
__global__ void k_pair_m2l(const PairJob *jobs, int njobs, int nbins, const uint32_t *bins, const uint32_t *bin_batch,
                           const uint32_t *d_nbatch, const PairEnt *list, const double *rot, int K, int p,
                           double2 *Y) {
  extern __shared__ __align__(16) double psm[];
  const int KI = K - (p + 1), R = K + KI, LD = R | 1;
  double *X = psm;                        // [R][PAIR_C]: real parts, then imaginary parts of m > 0
  double *W = X + (size_t)R * PAIR_C;     // [PAIR_KC][LD] operator columns
  int *hof = (int *)(W + (size_t)PAIR_KC * LD);  // [KI] half index of the ii-th m > 0 coefficient
  int *iof = hof + KI;                           // [K] position among the m > 0 coefficients or -1
  __shared__ PairEnt ent[PAIR_C];
  const uint32_t nb = *d_nbatch;
  for (int k = threadIdx.x; k < K; k += blockDim.x) {
    int n = 0;
    while ((n + 1) * (n + 2) / 2 <= k) ++n;
    const int m = k - n * (n + 1) / 2;
    const int ii = n * (n - 1) / 2 + m - 1;
    iof[k] = m ? ii : -1;
    if (m) hof[ii] = k;
  }
  const int r = threadIdx.x >> 1, cg = (threadIdx.x & 1) * (PAIR_C / 2);
  const bool im = r >= K;
  for (uint32_t b = blockIdx.x; b < nb; b += gridDim.x) {
    // last bin whose first batch is at or before b (empty bins share their successor's start)
    int lo = 0, hi = nbins - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (bin_batch[mid] <= b) lo = mid; else hi = mid - 1;
    }
    const int bin = lo;
    int jl = 0, jh = njobs - 1;
    while (jl < jh) {
      const int mid = (jl + jh + 1) >> 1;
      if (jobs[mid].bin0 <= bin) jl = mid; else jh = mid - 1;
    }
    const PairJob &J = jobs[jl];
    const int ct = bin - J.bin0, tau = ct % J.ntypes;
    const uint32_t first = (b - bin_batch[bin]) * PAIR_C;
    const int nc = (int)min((uint32_t)PAIR_C, bins[bin] - first);
    __syncthreads();
    if (threadIdx.x < PAIR_C)
      ent[threadIdx.x] = threadIdx.x < nc ? list[(size_t)b * PAIR_C + threadIdx.x] : PairEnt{0u, -1, 0};
    __syncthreads();
    for (int e = threadIdx.x; e < K * PAIR_C; e += blockDim.x) {
      const int c = e / K, k = e - c * K;
      const PairEnt en = ent[c];
      double vr = 0.0, vi = 0.0;
      if (en.s >= 0) {
        const int m = cK.mof[k];
        const double cs = rot[((size_t)en.o * (PMAX + 1) + m) * 2], sn = rot[((size_t)en.o * (PMAX + 1) + m) * 2 + 1];
        const double2 v = J.M[((size_t)en.s * J.ntypes + tau) * K + k];
        vr = cs * v.x - sn * v.y;
        vi = sn * v.x + cs * v.y;
      }
      X[k * PAIR_C + pair_pos(c)] = vr;
      if (iof[k] >= 0) X[(K + iof[k]) * PAIR_C + pair_pos(c)] = vi;
    }
    const double *P = J.ops + (size_t)ct * 2 * K * K, *Q = P + (size_t)K * K;
    double acc[PAIR_C / 2];
#pragma unroll
    for (int j = 0; j < PAIR_C / 2; ++j) acc[j] = 0.0;
    for (int k0 = 0; k0 < K; k0 += PAIR_KC) {
      __syncthreads();
      for (int e = threadIdx.x; e < R * PAIR_KC; e += blockDim.x) {
        const int row = e / PAIR_KC, kk = e % PAIR_KC, k = k0 + kk;
        double w = 0.0;
        if (row < K) {
          if (k < K) w = P[(size_t)row * K + k];
        } else if (k < KI) {
          w = Q[(size_t)hof[row - K] * K + hof[k]];
        }
        W[kk * LD + row] = w;
      }
      __syncthreads();
      const int kn = min(PAIR_KC, (im ? KI : K) - k0);
      if (r < R) {
        const double *xb = X + (size_t)((im ? K : 0) + k0) * PAIR_C + cg, *wb = W + r;
        switch ((nc + 1) >> 1) {  // columns of this thread (the last one empty for odd nc and the odd thread)
          case 1: pair_dot<1>(acc, wb, LD, xb, kn); break;
          case 2: pair_dot<2>(acc, wb, LD, xb, kn); break;
          case 3: pair_dot<3>(acc, wb, LD, xb, kn); break;
          default: pair_dot<4>(acc, wb, LD, xb, kn);
        }
      }
    }
    __syncthreads();
    if (r < R) {
#pragma unroll
      for (int j = 0; j < PAIR_C / 2; ++j) X[r * PAIR_C + cg + j] = acc[j];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < K * nc; e += blockDim.x) {
      const int c = e / K, k = e - c * K;
      const PairEnt en = ent[c];
      const int m = cK.mof[k];
      const double cs = rot[((size_t)en.o * (PMAX + 1) + m) * 2], sn = rot[((size_t)en.o * (PMAX + 1) + m) * 2 + 1];
      const double yr = X[k * PAIR_C + pair_pos(c)], yi = iof[k] >= 0 ? X[(K + iof[k]) * PAIR_C + pair_pos(c)] : 0.0;
      Y[(size_t)en.e * K + k] = make_double2(cs * yr + sn * yi, cs * yi - sn * yr);
    }
  }
}
static size_t pair_smem(int K, int p) {
  const int KI = K - (p + 1), R = K + KI;
  return sizeof(double) * ((size_t)R * PAIR_C + (size_t)PAIR_KC * (R | 1)) + sizeof(int) * (KI + K);
}

// L[t] += the slots of target t in the window, in slot order: one CTA per target, the slot range in
// PAIR_PARTS contiguous parts summed side by side and added in order.  Free-space and reaction jobs
// of one level add into the same expansions: g0 selects one kind per launch.
constexpr int PAIR_PARTS = 4;
__global__ void k_pair_sum(const PairJob *jobs, int njobs, int64_t g0, const uint32_t *e0, const uint32_t *cnt, uint32_t w0,
                           uint32_t w1, const double2 *Y, int K) {
  __shared__ double2 part[PAIR_PARTS][KHALF_MAX];
  const int64_t g = g0 + blockIdx.x;
  const uint32_t a = max(e0[g], w0), z = min(e0[g] + cnt[g], w1);
  if (a >= z) return;
  const PairJob &J = jobs[pair_find_job(jobs, njobs, g)];
  const uint32_t len = (z - a + PAIR_PARTS - 1) / PAIR_PARTS;
  for (int i = threadIdx.x; i < PAIR_PARTS * K; i += blockDim.x) {
    const int q = i / K, k = i - q * K;
    const uint32_t b0 = a + q * len, b1 = min(b0 + len, z);
    double sx = 0.0, sy = 0.0;
#pragma unroll 4
    for (uint32_t e = b0; e < b1; ++e) {
      const double2 v = Y[(size_t)(e - w0) * K + k];
      sx += v.x;
      sy += v.y;
    }
    part[q][k] = make_double2(sx, sy);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < K; k += blockDim.x) {
    double2 &d = J.L[(size_t)(g - J.t0) * K + k];
    double sx = 0.0, sy = 0.0;
#pragma unroll
    for (int q = 0; q < PAIR_PARTS; ++q) {
      sx += part[q][k].x;
      sy += part[q][k].y;
    }
    d.x += sx;
    d.y += sy;
  }
}

// every FP64 translation of the jobs (free-space jobs first; t0, bin0 filled in here)
static void launch_pair_m2l_part(Ctx &c, std::vector<PairJob> &jobs, const std::vector<int> &ncls, const double *rot) {
  int64_t ntot = 0, nfree = 0;
  int nbins = 0;
  for (size_t k = 0; k < jobs.size(); ++k) {
    jobs[k].t0 = ntot;
    jobs[k].bin0 = nbins;
    ntot += jobs[k].ntb;
    if (!jobs[k].ktrow) nfree = ntot;
    nbins += ncls[k] * jobs[k].ntypes;
  }
  if (!ntot) return;
  const int nj = (int)jobs.size(), K = c.K;
  PairJob *dj = c.arena.get<PairJob>(jobs.size());
  LPB_CUDA(cudaMemcpyAsync(dj, jobs.data(), sizeof(PairJob) * jobs.size(), cudaMemcpyHostToDevice, c.stream));
  uint32_t *cnt = c.arena.get<uint32_t>(ntot), *e0 = c.arena.get<uint32_t>(ntot);
  uint32_t *d_tot = c.arena.get<uint32_t>(2);
  const unsigned wb = (unsigned)((ntot + 3) / 4);
  k_pair_walk<0><<<wb, 128, 0, c.stream>>>(dj, nj, ntot, cnt, nullptr, 0, 0, nullptr, nullptr, nullptr);
  LPB_LAUNCH();
  c.launches++;
  scan_u32(c, cnt, e0, ntot, d_tot);
  uint32_t *h = (uint32_t *)c.h_pinned;
  LPB_CUDA(cudaMemcpyAsync(h, d_tot, sizeof(uint32_t), cudaMemcpyDeviceToHost, c.stream));
  LPB_CUDA(cudaStreamSynchronize(c.stream));
  const uint64_t total = h[0];
  if (!total) return;
  uint32_t *bins = c.arena.get<uint32_t>(nbins), *nbt = c.arena.get<uint32_t>(nbins),
           *bb = c.arena.get<uint32_t>(nbins), *cur = c.arena.get<uint32_t>(nbins);
  uint64_t win = std::min<uint64_t>(total, std::max<uint64_t>(c.pair_window / (sizeof(double2) * K), 1));
  double2 *Y = nullptr;
  PairEnt *list = nullptr;
  for (const Arena::Mark mark = c.arena.mark(); !list;) {  // smaller windows where memory is short
    try {
      Y = c.arena.get<double2>((size_t)win * K);
      list = c.arena.get<PairEnt>((size_t)win + (size_t)nbins * PAIR_C);
    } catch (const StatusError &) {
      if (win <= PAIR_WINDOW_MIN) throw;
      c.arena.rewind(mark);
      win = (win + 1) / 2;
    }
  }
  const int R = 2 * K - (c.p + 1), threads = (2 * R + 31) / 32 * 32;
  LPB_ATTR_ONCE(k_pair_m2l, pair_smem(KHALF_MAX, PMAX));
  for (uint64_t w0 = 0; w0 < total; w0 += win) {
    const uint32_t a = (uint32_t)w0, z = (uint32_t)std::min<uint64_t>(w0 + win, total);
    LPB_CUDA(cudaMemsetAsync(bins, 0, sizeof(uint32_t) * nbins, c.stream));
    LPB_CUDA(cudaMemsetAsync(cur, 0, sizeof(uint32_t) * nbins, c.stream));
    k_pair_walk<1><<<wb, 128, 0, c.stream>>>(dj, nj, ntot, cnt, e0, a, z, bins, nullptr, nullptr);
    LPB_LAUNCH();
    k_pair_batches<<<(unsigned)((nbins + 255) / 256), 256, 0, c.stream>>>(bins, nbins, nbt);
    LPB_LAUNCH();
    scan_u32(c, nbt, bb, nbins, d_tot + 1);
    k_pair_walk<2><<<wb, 128, 0, c.stream>>>(dj, nj, ntot, cnt, e0, a, z, cur, bb, list);
    LPB_LAUNCH();
    // at most one batch per PAIR_C translations and one partial batch per bin; idle CTAs return
    const uint64_t nb = std::min<uint64_t>((uint64_t)(z - a) / PAIR_C + nbins, 1 << 20);
    k_pair_m2l<<<(unsigned)nb, threads, pair_smem(K, c.p), c.stream>>>(dj, nj, nbins, bins, bb, d_tot + 1, list, rot, K,
                                                                        c.p, Y);
    LPB_LAUNCH();
    c.launches += 4;
    for (int64_t g0 = 0; g0 < ntot; g0 = nfree > g0 ? nfree : ntot) {
      const int64_t n = (nfree > g0 ? nfree : ntot) - g0;
      k_pair_sum<<<(unsigned)n, 256, 0, c.stream>>>(dj, nj, g0, e0, cnt, a, z, Y, K);
      LPB_LAUNCH();
      c.launches++;
    }
  }
}

// the jobs in parts of at most pair_part translations (their numbers are 32-bit), whole targets each, in the jobs' order,
// so that a target's free-space and reaction sums are added as in one part
static void launch_pair_m2l(Ctx &c, const std::vector<PairJob> &jobs, const std::vector<int> &ncls, const double *rot) {
  std::vector<PairJob> part;
  std::vector<int> pcls;
  uint64_t room = c.pair_part;
  const Arena::Mark mark = c.arena.mark();  // a part follows the one before it in stream order, in its memory
  for (size_t k = 0; k < jobs.size(); ++k) {
    const PairJob &J = jobs[k];
    const uint64_t per = (uint64_t)NOFF * J.ntypes;  // at most, per target
    for (int32_t t = 0; t < J.ntb;) {
      if (room < per) {
        launch_pair_m2l_part(c, part, pcls, rot);
        c.arena.rewind(mark);
        part.clear();
        pcls.clear();
        room = c.pair_part;
      }
      const int32_t n = (int32_t)std::min<uint64_t>((uint64_t)(J.ntb - t), room / per);
      PairJob p = J;
      p.vlist += (size_t)t * NOFF;
      if (p.ktrow) p.ktrow += t;
      p.L += (size_t)t * c.K;
      p.ntb = n;
      part.push_back(p);
      pcls.push_back(ncls[k]);
      room -= per * (uint64_t)n;
      t += n;
    }
  }
  launch_pair_m2l_part(c, part, pcls, rot);
  c.arena.rewind(mark);  // what follows on this stream may take the slots' memory
}
