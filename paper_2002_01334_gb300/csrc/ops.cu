// Translation operators, built on the device in FP64 for every evaluation.
//
// All translations have the azimuth-factored form (half representation m >= 0):
//   X'_{nu mu} = e^{i mu phi} X_{nu mu},  Y_{nm} = P Re X' + i Q Im X',  out_{nm} += e^{-i m phi} Y_{nm}
// with real P, Q of size K x K, K = (p+1)(p+2)/2.
//  * free-space M2M / L2L / M2L (Sec. 3.1, Theorems 1-3): Gaunt-coefficient sums over
//    i_q(lambda b) or k_q(lambda b) times Phat_q(cos theta_b);
//  * reaction M2L (Sec. 3.4 eq. metoleimage2, Sec. 3.5): the scaled Sommerfeld integrals
//    S^K S_{K d, ij} (eq. M2Ltable) by composite Gauss-Legendre quadrature for d = 0, 1,
//    the forward recurrence (eq. recurrence1) for d >= 2, and a Legendre-product expansion
//    of the two plane-wave factors (eq. metoletableform), in this library's own derivation.
// Scaling (Sec. 3.5, the rescaled expansions): with h the box size, multipole coefficients are stored as
// M~_n = M_n (2n+1)!!/(lambda h)^n and local ones as L~_n = c L_n (lambda h)^n/(2n+1)!!
// (c = lambda/(2 pi^2 eps) for the free-space part, 1 for reaction parts), so that
// phi = sum L~_nm itilde_n(lambda r) R_n^m(r/h) with R_n^m = r^n Y_n^m.
#include "internal.h"

#include <mutex>

namespace lpb {

struct OpDesc {
  int kind;     // 0 = M2L free, 1 = M2M, 2 = L2L
  int out_inv;  // 0: out scale x^n/(2n+1)!!, 1: (2n+1)!!/x^n
  int in_inv;
  int dir;      // direction of b: free M2L class (< NFREE_CLS), NFREE_CLS + cz for M2M / L2L (Ctx::phat_dir)
  double lam, bnorm, cosb, xout, xin, pref;
  int64_t dst;  // element offset of P (Q follows after K*K)
};

// half-representation index o = n(n+1)/2 + m -> (n, m), integer arithmetic only
__device__ __forceinline__ void hdecode(int o, int &n, int &m) {
  n = 0;
  while ((n + 1) * (n + 2) / 2 <= o) ++n;
  m = o - n * (n + 1) / 2;
}

// Per-descriptor radial factors, one thread each: f[q] = k_q or i_q (lambda |b|) and the
// output / input scalings so[n], si[n], stored as [NPREP] doubles per descriptor.  The angular
// factor Phat_q^k(cos theta_b) depends only on the direction of b and comes from Ctx::phat_dir.
constexpr int PREP_F = 0, PREP_SO = 2 * PMAX + 1, PREP_SI = PREP_SO + PMAX + 1, NPREP = PREP_SI + PMAX + 1;
constexpr int NPL_MAX = (2 * PMAX + 1) * (2 * PMAX + 2) / 2;

__global__ void k_ops_prep(const OpDesc *descs, int nd, int p, double *prep) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nd) return;
  const OpDesc d = descs[i];
  double *w = prep + (size_t)i * NPREP;
  const int qmax = 2 * p;
  const double x = d.lam * d.bnorm;
  if (d.kind == 0) kbessel_all(x, qmax, w + PREP_F);
  else ibessel_all(x, qmax, w + PREP_F);
  double a = 1.0, b = 1.0;  // x^n / (2n+1)!!
  for (int n = 0; n <= p; ++n) {
    if (n > 0) {
      a *= d.xout / (2.0 * n + 1.0);
      b *= d.xin / (2.0 * n + 1.0);
    }
    w[PREP_SO + n] = (d.out_inv ? 1.0 / a : a) * d.pref;
    w[PREP_SI + n] = d.in_inv ? 1.0 / b : b;
  }
}

constexpr int OPS_SPLIT = 4;  // CTAs per descriptor

// Bound: the FP64 pipe (0.63 T FMA/s).  All three kinds are the same sum over q of
// f_q Phat_q^{mu'-m} G(n, m; nu, mu'; q), mu' = +-mu: the product f_q Phat_q^k is formed once per
// descriptor, so a term is one FMA (three FP64 operations before: 0.25 ms per free-space group at p = 10,
// three levels), and the table is read with the column index fastest, so that a warp's loads
// coalesce.
template <typename T>
__global__ void k_build_ops(const OpDesc *descs, const double *prep, const double *phat_dir, int p, int K,
                            const double *gaunt, T *out) {
  const OpDesc d = descs[blockIdx.x];
  __shared__ double w[NPREP], Pl[NPL_MAX];
  const double *pw = prep + (size_t)blockIdx.x * NPREP;
  for (int e = threadIdx.x; e < NPREP; e += blockDim.x) w[e] = pw[e];
  __syncthreads();
  const double *so = w + PREP_SO, *si = w + PREP_SI;
  const int qmax = 2 * p, npl = (qmax + 1) * (qmax + 2) / 2;
  const double *pd = phat_dir + (size_t)d.dir * npl;
  for (int e = threadIdx.x; e < npl; e += blockDim.x) {
    int q, k;
    hdecode(e, q, k);
    Pl[e] = w[PREP_F + q] * pd[e];
  }
  __syncthreads();
  const int NF = (p + 1) * (p + 1), NQ = 2 * p + 1;
  for (int e = blockIdx.y * blockDim.x + threadIdx.x; e < K * K; e += gridDim.y * blockDim.x) {
    const int o = e / K, i = e % K;
    int n, m, nu, mu;
    hdecode(o, n, m);
    hdecode(i, nu, mu);
    double r[2] = {0.0, 0.0};
    const double *G = gaunt + (size_t)fidx(n, m) * NQ * NF;
    const double sc = 4.0 * PI * so[n] * si[nu];
    for (int sgn = 0; sgn < 2; ++sgn) {
      const int mus = sgn ? -mu : mu;
      if (sgn && mu == 0) break;
      const int k = mus - m, ak = k < 0 ? -k : k;
      int q0 = n > nu ? n - nu : nu - n;
      if (q0 < ak) q0 = ak + ((n + nu + ak) & 1);
      double acc = 0.0;
      for (int q = q0; q <= n + nu; q += 2) acc = fma(Pl[hidx(q, ak)], G[(size_t)q * NF + fidx(nu, mus)], acc);
      const bool neg = (k < 0 && (ak & 1)) != (d.kind == 0 && (n & 1));  // Phat_q^{-k} = (-1)^k Phat_q^k
      r[sgn] = neg ? -acc * sc : acc * sc;
    }
    double P, Q;
    if (mu == 0) { P = r[0]; Q = 0.0; }
    else {
      const double r1 = (mu & 1) ? -r[1] : r[1];
      P = r[0] + r1;
      Q = r[0] - r1;
    }
    // M2L operators row by row; M2M and L2L with the output row fastest (their kernels own a row per thread)
    const size_t at = d.dst + (d.kind == 0 ? (size_t)o * K + i : (size_t)i * K + o);
    out[at] = (T)P;
    out[at + (size_t)K * K] = (T)Q;
  }
}

// ---------------------------------------------------------------------------------------
// Reaction operators
// ---------------------------------------------------------------------------------------
constexpr int MAXPANEL = 1024;

__device__ __forceinline__ int stab_index(int KT, int K, int d, int ij) { return ((K * (KT + 1)) + d) * 4 + ij; }

// panels of width at most wmax, graded towards u = 0: at most grow (lmin + u)
__device__ void make_panels(double umax, double wmax, double lmin, double grow, double *pu, double *pw, int *np) {
  int n = 0;
  double u = 0.0;
  while (u < umax && n < MAXPANEL) {
    double w = fmin(wmax, grow * (lmin + u));
    if (u + w > umax) w = umax - u;
    pu[n] = u;
    pw[n] = w;
    u += w;
    ++n;
  }
  *np = n;
}

// Gauss-Legendre rules on [-1,1] (nodes by Newton iteration on the host): 32 points for the Sommerfeld
// tables, 16 for the reaction near field
constexpr int GLN = 32;
__constant__ double c_glx[16], c_glw[16], c_gl32x[GLN], c_gl32w[GLN];
static std::atomic<uint64_t> g_gl_ready{0};
static void gl_rule(int n, double *x, double *w) {
  for (int i = 0; i < n; ++i) {
    long double z = cosl(3.14159265358979323846264338L * (i + 0.75L) / (n + 0.5L)), dp = 1;
    for (int it = 0; it < 100; ++it) {
      long double p0 = 1, p1 = z;
      for (int k = 2; k <= n; ++k) { long double p2 = ((2 * k - 1) * z * p1 - (k - 1) * p0) / k; p0 = p1; p1 = p2; }
      dp = n * (z * p1 - p0) / (z * z - 1);
      const long double dz = p1 / dp;
      z -= dz;
      if (fabsl(dz) < 1e-19L) break;
    }
    long double p0 = 1, p1 = z;
    for (int k = 2; k <= n; ++k) { long double p2 = ((2 * k - 1) * z * p1 - (k - 1) * p0) / k; p0 = p1; p1 = p2; }
    dp = n * (z * p1 - p0) / (z * z - 1);
    x[i] = (double)z;
    w[i] = (double)(2 / ((1 - z * z) * dp * dp));
  }
}
void upload_gl() {
  if (!not_done_on_device(g_gl_ready)) return;
  double x[GLN], w[GLN];
  gl_rule(16, x, w);
  LPB_CUDA(cudaMemcpyToSymbol(c_glx, x, sizeof(double) * 16));
  LPB_CUDA(cudaMemcpyToSymbol(c_glw, w, sizeof(double) * 16));
  gl_rule(GLN, x, w);
  LPB_CUDA(cudaMemcpyToSymbol(c_gl32x, x, sizeof x));
  LPB_CUDA(cudaMemcpyToSymbol(c_gl32w, w, sizeof w));
  mark_done_on_device(g_gl_ready);
}
__device__ __forceinline__ void gl16(double *x, double *w) {
  for (int i = 0; i < 16; ++i) { x[i] = c_glx[i]; w[i] = c_glw[i]; }
}

// Quadrature of S^K S_{K d, ij} for d = 0, 1, K = 0..KT on one composite Gauss-Legendre node
// set per (component, level) in u = lambda_rho h: panel width min(6, 3 (Lambda_min + u)), graded near
// u = 0 to resolve the branch points at u = +-i Lambda.  Node data (k_stab_nodes):
//   nd[q] = {u, w sigma / u_z, Lam / u_z, Lamp / u'_z, e^{-u_z (k+1/2)} (k < NKT),
//            e^{-u'_z (k+1/2)} (k < NKT)}
// and, shared by every descriptor on the node set, bes[q] = {J0(u rho_r), J1(u rho_r) (r < NRHO)}.
constexpr int ND_ET = 4, ND_ES = ND_ET + NKT, NDF = ND_ES + NKT, NBES = 2 * NRHO;
constexpr double ST_WMAX = 6.0, ST_GROW = 3.0;

// host: the u beyond which u^KT e^{-zeta u} has fallen by tol (and e^-3 more) below its peak
// at u = KT/zeta
static double node_umax(int KT, double zeta, double tol) {
  const double pk = fmax(KT / zeta, 1.0 / zeta);
  const double target = KT * log(pk) - zeta * pk + log(tol) - 3.0;
  double umax = pk;
  while (KT * log(umax) - zeta * umax > target) umax += 0.25 / zeta;
  return umax;
}

struct NDesc {
  double umax, wmax, lmin;
  double ucut[NKT];  // truncation point for zeta = k_t + k_s + 1 = 1 .. NKT
  int npan, nq;
  double *nodes;        // [nq][NDF]
  const double *bes;    // [nq][NBES]
};

// J0(u rho_r), J1(u rho_r) at the nodes of one node set, shared by every descriptor using it
__global__ void k_stab_bessel(NDesc N, double *bes) {
  __shared__ double pu[MAXPANEL], pw[MAXPANEL];
  __shared__ int npan;
  if (threadIdx.x == 0) make_panels(N.umax, N.wmax, N.lmin, ST_GROW, pu, pw, &npan);
  __syncthreads();
  // one thread per (node, rho value): the node set is short, so a thread per node alone would
  // leave most of the GPU idle
  const int64_t total = (int64_t)N.nq * NRHO;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int j = (int)(e / NRHO), r = (int)(e % NRHO);
    double *o = bes + (size_t)j * NBES;
    if (j >= npan * GLN) {
      o[r] = 0.0;
      o[NRHO + r] = 0.0;
      continue;
    }
    const int pi_ = j / GLN, gi = GLN - 1 - (j % GLN);  // ascending abscissae
    const double u = pu[pi_] + 0.5 * pw[pi_] * (c_gl32x[gi] + 1.0);
    const double x = u * sqrt((double)rho2_of(r));
    o[r] = j0(x);
    o[NRHO + r] = j1(x);
  }
}

__global__ void k_stab_nodes(const RDesc *descs, const NDesc *nds, Medium md) {
  const RDesc D = descs[blockIdx.y];
  const NDesc N = nds[blockIdx.y];
  __shared__ double pu[MAXPANEL], pw[MAXPANEL];
  __shared__ int npan;
  if (threadIdx.x == 0) make_panels(N.umax, N.wmax, N.lmin, ST_GROW, pu, pw, &npan);
  __syncthreads();
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < N.nq; j += gridDim.x * blockDim.x) {
    double *o = N.nodes + (size_t)j * NDF;
    if (j >= npan * GLN) {
      for (int k = 0; k < NDF; ++k) o[k] = 0.0;
      continue;
    }
    const int pi_ = j / GLN, gi = GLN - 1 - (j % GLN);  // ascending abscissae
    const double u = pu[pi_] + 0.5 * pw[pi_] * (c_gl32x[gi] + 1.0);
    const double w = 0.5 * pw[pi_] * c_gl32w[gi];
    const double sg = layer_sigma(md, u / D.h, D.l, D.a, D.lp, D.b);
    const double uz = sqrt(D.Lam * D.Lam + u * u), uzp = sqrt(D.Lamp * D.Lamp + u * u);
    o[0] = u;
    o[1] = w * sg / uz;
    o[2] = D.Lam / uz;
    o[3] = D.Lamp / uzp;
    for (int k = 0; k < NKT; ++k) {
      o[ND_ET + k] = exp(-uz * (k + 0.5));
      o[ND_ES + k] = exp(-uzp * (k + 0.5));
    }
  }
}

// a_n = sqrt(n (n+1)) and 1/a_n for n <= 2 KMAX_TAB + 1 (host, long double), for the recurrence
__constant__ double c_an[2 * KMAX_TAB + 2], c_ian[2 * KMAX_TAB + 2];
static std::atomic<uint64_t> g_an_ready{0};
void upload_an() {
  if (!not_done_on_device(g_an_ready)) return;
  double a[2 * KMAX_TAB + 2], ia[2 * KMAX_TAB + 2];
  for (int n = 0; n < 2 * KMAX_TAB + 2; ++n) {
    const long double v = sqrtl((long double)n * (n + 1));
    a[n] = (double)v;
    ia[n] = n ? (double)(1.0L / v) : 0.0;
  }
  LPB_CUDA(cudaMemcpyToSymbol(c_an, a, sizeof a));
  LPB_CUDA(cudaMemcpyToSymbol(c_ian, ia, sizeof ia));
  mark_done_on_device(g_an_ready);
}

// Tables of ST_NC classes with one (k_t, k_s) and consecutive rho per CTA: the d = 0, 1 columns by quadrature,
// then the forward recurrence in d (Sec. 3.5 eq. recurrence1),
//   S_{K,d+1} = (2d / a_{K+d}) (1/rho) S_{K-1,d} - (a_{K-d} / a_{K+d}) S_{K,d-1}.
// Only the entries with K - d odd are formed: the operators use no others, because
// K = 1 + |m| + |mu| + 2s and d = |mu - m| differ by an odd number (and the recurrence stays among them).
// Quadrature: per chunk of ST_CH nodes the power columns u^K and, per class, the eight node values
// v_{d,ij} = w sigma/u_z (Lam/u_z)^i (Lamp/u'_z)^j Z_{kt,ks} J_d(u rho) are staged in shared memory; thread
// (class, d, i, j, K) accumulates sum_q u_q^K v_{d,ij}(q), a [KT+1 x Q] x [Q x 8] product.
// Bound: the FP64 pipe (86 % busy with one class per CTA and 16-point panels of width 2: 0.26 ms a group
// at p = 10).  So: the powers once for four classes, nodes beyond the class's cut not at all, and 32-point
// panels of width 6, which need a third fewer nodes: with |zeta + i rho| <= 8.7 the rule's error on a
// panel is (e omega / 128)^64, omega <= 26, ~1e-17 of the integrand's scale (16 points on width 2: 1e-14);
// towards u = 0, panels of 3 (Lambda + u) with the branch points at +-i Lambda: below 1e-20.
constexpr int ST_NC = 4, ST_CH = 128, ST_LD = ST_CH + 1, ST_THREADS = 384, ST_NOUT = 2;
static_assert(NRHO % ST_NC == 0, "classes of a CTA share (k_t, k_s)");
static_assert(4 * KMAX_TAB * ST_NC <= ST_NOUT * ST_THREADS, "outputs per thread");
__global__ void __launch_bounds__(ST_THREADS) k_stab_table(const RDesc *descs, const NDesc *nds, int KT,
                                                           const double *sfac) {
  const RDesc D = descs[blockIdx.y];
  const NDesc N = nds[blockIdx.y];
  const int kk = blockIdx.x / (NRHO / ST_NC), ri0 = (blockIdx.x % (NRHO / ST_NC)) * ST_NC;
  unsigned use = 0;
  for (int r = 0; r < ST_NC; ++r)
    if (!D.used || D.used[(ri0 + r) * NKK + kk]) use |= 1u << r;
  if (!use) return;
  extern __shared__ double stsm[];
  double *Pw = stsm;                               // [KT+1][ST_LD] powers
  double *V = Pw + (size_t)(KT + 1) * ST_LD;       // [ST_NC][8][ST_LD] node values
  double *col = V + (size_t)ST_NC * 8 * ST_LD;     // [3][ST_NC][(KT+1) 4] columns d - 1, d, d + 1
  const int cl = (KT + 1) * 4;
  int kt, ks;
  kk_decode(kk, kt, ks);
  const double ucut = N.ucut[kt + ks];
  const int tid = threadIdx.x;
  // outputs of this thread: class, d, ij, K with K - d odd
  const int n0 = (KT + 1) / 2, n1 = KT / 2;  // K odd (d = 0): 1,3,..; K even >= 2 (d = 1): 2,4,..
  const int nout = 4 * (n0 + n1);
  int orr[ST_NOUT], od[ST_NOUT], oij[ST_NOUT], oK[ST_NOUT];
  double acc[ST_NOUT];
#pragma unroll
  for (int x = 0; x < ST_NOUT; ++x) {
    const int t = tid + x * ST_THREADS;
    acc[x] = 0.0;
    oK[x] = -1;
    orr[x] = od[x] = oij[x] = 0;
    if (t < nout * ST_NC && ((use >> (t / nout)) & 1u)) {
      orr[x] = t / nout;
      const int o = t % nout, k = o >> 2;
      oij[x] = o & 3;
      od[x] = k < n0 ? 0 : 1;
      oK[x] = k < n0 ? 2 * k + 1 : 2 * (k - n0) + 2;
    }
  }
  for (int c0 = 0; c0 < N.nq; c0 += ST_CH) {
    bool in = false;
    if (tid < ST_CH && c0 + tid < N.nq) {
      const double u = N.nodes[(size_t)(c0 + tid) * NDF];
      in = u <= ucut && u > 0.0;
      if (in) {
        double pw = u;
        for (int K = 1; K <= KT; ++K) {
          Pw[K * ST_LD + tid] = pw;
          pw *= u;
        }
      }
    }
    const int nn = __syncthreads_count(in);  // the nodes ascend: those within the cut come first
    for (int e = tid; e < ST_NC * ST_CH; e += ST_THREADS) {
      const int r = e / ST_CH, j = e % ST_CH;
      if (j >= nn || !((use >> r) & 1u)) continue;
      const double *o = N.nodes + (size_t)(c0 + j) * NDF, *bs = N.bes + (size_t)(c0 + j) * NBES + ri0 + r;
      const double base = o[1] * o[ND_ET + kt] * o[ND_ES + ks], fi = o[2], fj = o[3], ff = fi * fj;
      const double b0 = base * bs[0], b1 = base * bs[NRHO];
      double *v = V + (size_t)r * 8 * ST_LD + j;
      v[0 * ST_LD] = b0;
      v[1 * ST_LD] = b0 * fj;
      v[2 * ST_LD] = b0 * fi;
      v[3 * ST_LD] = b0 * ff;
      v[4 * ST_LD] = b1;
      v[5 * ST_LD] = b1 * fj;
      v[6 * ST_LD] = b1 * fi;
      v[7 * ST_LD] = b1 * ff;
    }
    __syncthreads();
#pragma unroll
    for (int x = 0; x < ST_NOUT; ++x)
      if (oK[x] >= 0) {
        const double *pr = Pw + oK[x] * ST_LD, *vr = V + (orr[x] * 8 + od[x] * 4 + oij[x]) * ST_LD;
        double a = acc[x];
        for (int j = 0; j < nn; ++j) a = fma(pr[j], vr[j], a);
        acc[x] = a;
      }
    __syncthreads();
    if (nn < ST_CH) break;
  }
  const size_t TS = (size_t)(KT + 1) * (KT + 1) * 4;
  auto table = [&](int r) {
    return D.stab + ((size_t)((ri0 + r) * NKK + kk - D.cls0) * D.ntypes + D.tau) * TS;
  };
#pragma unroll
  for (int x = 0; x < ST_NOUT; ++x)
    if (oK[x] >= 0) {
      const double v = acc[x] * (1.0 / sfac[oK[x] * (KMAX_TAB + 1) + od[x]]);
      table(orr[x])[stab_index(KT, oK[x], od[x], oij[x])] = v;
      col[(od[x] * ST_NC + orr[x]) * cl + oK[x] * 4 + oij[x]] = v;
    }
  __syncthreads();
  for (int d = 1; d < KT; ++d) {
    const int per = 4 * ((KT - d) / 2);  // K = d + 2, d + 4, ...
    const double *c1 = col + (d % 3) * ST_NC * cl, *c0 = col + ((d - 1) % 3) * ST_NC * cl;
    double *c2 = col + ((d + 1) % 3) * ST_NC * cl;
    for (int e = tid; e < per * ST_NC; e += ST_THREADS) {
      const int r = e / per, x = e % per, K = d + 2 + 2 * (x >> 2), ij = x & 3;
      if (!((use >> r) & 1u)) continue;
      const double rh = sqrt((double)rho2_of(ri0 + r));
      double v = 0.0;
      if (rh > 0.0) {
        const double ia = c_ian[K + d];
        v = (2.0 * d * ia * (1.0 / rh)) * c1[r * cl + (K - 1) * 4 + ij] - (c_an[K - d] * ia) * c0[r * cl + K * 4 + ij];
      }
      c2[r * cl + K * 4 + ij] = v;
      table(r)[stab_index(KT, K, d + 1, ij)] = v;
    }
    __syncthreads();
  }
}
static size_t stab_table_smem(int KT) {
  return sizeof(double) * ((size_t)(KT + 1 + ST_NC * 8) * ST_LD + (size_t)3 * ST_NC * (KT + 1) * 4);
}

// host: node set of one (component, level) covering every class (zeta >= 1, rho <= sqrt(50) h)
// number of panels of the graded rule (host mirror of make_panels)
static int count_panels(double umax, double wmax, double lmin, double grow) {
  int n = 0;
  double u = 0.0;
  while (u < umax && n < MAXPANEL) {
    double w = fmin(wmax, grow * (lmin + u));
    if (u + w > umax) w = umax - u;
    u += w;
    ++n;
  }
  return n;
}

static NDesc node_desc(int KT, double tol, double Lam, double Lamp) {
  NDesc N;
  N.umax = node_umax(KT, 1.0, tol);
  for (int z = 0; z < NKT; ++z) N.ucut[z] = node_umax(KT, z + 1.0, tol);
  N.wmax = ST_WMAX;
  N.lmin = fmin(Lam, Lamp);
  N.npan = count_panels(N.umax, N.wmax, N.lmin, ST_GROW);
  N.nq = N.npan * GLN;
  N.nodes = nullptr;
  N.bes = nullptr;
  return N;
}

// C_s(n,m,nu,mu) = sum_{k+k'=s} c^{nm}_k c^{nu mu}_{k'} Lam^{n-m-2k} Lamp^{nu-mu-2k'}, s <= (n-m+1)/2 + (nu-mu+1)/2
// (the assembly reads no others).  Bound: the FP64 pipe, so the powers go into the two factors once per CTA and
// a term is one FMA (four FP64 operations before): 0.110 -> 0.040 ms at p = 10, 0.57 -> 0.20 ms for four layers at p = 12.
__global__ void k_react_coef(const RDesc *descs, const double *tpoly, int tpk, int p, int K) {
  const RDesc D = descs[blockIdx.y];
  __shared__ double pl[2][PMAX + 3];  // Lam^e, Lamp^e for e = -1..p+1 at index e+1
  extern __shared__ double coef_sm[];
  double *A = coef_sm, *B = A + (size_t)K * tpk;  // c^{nm}_k Lam^{n-m-2k}, c^{nu mu}_k Lamp^{nu-mu-2k}
  if (threadIdx.x < 2) {
    const double v = threadIdx.x ? D.Lamp : D.Lam;
    double *t = pl[threadIdx.x];
    t[0] = 1.0 / v;
    t[1] = 1.0;
    for (int e = 2; e <= p + 2; ++e) t[e] = t[e - 1] * v;
  }
  __syncthreads();
  for (int x = threadIdx.x; x < K * tpk; x += blockDim.x) {
    const int o = x / tpk, k = x % tpk;
    int n, m;
    hdecode(o, n, m);
    const int e = n - m - 2 * k + 1;
    const double c = e >= 0 ? tpoly[x] : 0.0;
    A[x] = e >= 0 ? c * pl[0][e] : 0.0;
    B[x] = e >= 0 ? c * pl[1][e] : 0.0;
  }
  __syncthreads();
  const int NS = p + 2;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= K * K) return;
  const int o = e / K, i = e % K;
  int n, m, nu, mu;
  hdecode(o, n, m);
  hdecode(i, nu, mu);
  const int k1 = (n - m + 1) / 2, k2 = (nu - mu + 1) / 2;
  const double *a = A + o * tpk, *b = B + i * tpk;
  for (int s = 0; s <= k1 + k2; ++s) {
    double acc = 0.0;
    for (int k = max(0, s - k2); k <= min(k1, s); ++k) acc = fma(a[k], b[s - k], acc);
    const float h = (float)acc;
    D.coef[(size_t)e * NS + s] = make_float2(h, (float)(acc - (double)h));
  }
}

// double-float arithmetic (value = hi + lo, two FP32 numbers; about 44 significant bits) on
// the FP32 pipes: exact products by FMA, sums by the two-sum of Knuth, whose error joins the low part.  The
// two parts of a sum are not renormalised on the way (the two-sum asks for no order of its operands, the low
// part stays a few ulps of the partial sums): 12 operations a term instead of 15, assembly 0.77 -> 0.73 ms at p = 10.
// The _rn intrinsics keep the compiler from contracting the error-free transformations.
__device__ __forceinline__ float2 df_split(double v) {
  const float h = (float)v;
  return make_float2(h, (float)(v - (double)h));
}
// hi + lo of (a.hi + a.lo) + (b.hi + b.lo) rounded to one FP32 number, without losing the low parts
// to cancellation between a and b
__device__ __forceinline__ float df_sum_f(float2 a, float2 b) {
  const float s = __fadd_rn(a.x, b.x);
  const float v = __fsub_rn(s, a.x);
  const float e = __fadd_rn(__fsub_rn(a.x, __fsub_rn(s, v)), __fsub_rn(b.x, v));
  return __fadd_rn(s, __fadd_rn(e, __fadd_rn(a.y, b.y)));
}
__device__ __forceinline__ void df_fma(float2 a, float2 b, float2 &acc) {
  const float p = __fmul_rn(a.x, b.x);
  float e = fmaf(a.x, b.x, -p);  // rounding error of p, exactly
  e = fmaf(a.x, b.y, e);
  e = fmaf(a.y, b.x, e);
  const float s = __fadd_rn(acc.x, p);
  const float v = __fsub_rn(s, acc.x);
  const float t = __fadd_rn(__fsub_rn(acc.x, __fsub_rn(s, v)), __fsub_rn(p, v));
  acc = make_float2(s, __fadd_rn(t, __fadd_rn(acc.y, e)));
}

// ASM_CC classes per CTA share each entry's decode and coefficient loads.  The tables sit in shared memory by
// (d, t), K = d + 1 + 2t (the entries with K - d odd, no others are read), a quarter of the square
// [K][d] array, so that six CTAs fit an SM instead of three; rows are padded to an odd number of records.
// Every level and type of every group in one launch: the levels one after another (300 CTAs each) left
// most of the GPU idle (0.11 ms a level, 1.55 ms in all at p = 10).
constexpr int ASM_CC = 4;
LPB_HD int asm_row(int KT) { return (KT + 1) / 2 * 4 + 1; }
LPB_HD int asm_size(int p, int KT) { return (2 * p + 1) * asm_row(KT); }
template <typename T>
__global__ void k_react_assemble(const RDesc *descs, int p, int K, int KT, const double *sfac) {
  const RDesc D = descs[blockIdx.y];
  const int cls0 = blockIdx.x * ASM_CC;
  extern __shared__ double asm_sm[];
  const size_t TS = (size_t)(KT + 1) * (KT + 1) * 4;
  const int AR = asm_row(KT), AS = asm_size(p, KT), NT = (KT + 1) / 2;
  float2 *Sf = (float2 *)asm_sm;  // [ASM_CC][AS]: sqrt((K+d)!(K-d)!) S^K S_{K d, ij}, double-float
  T *out = (T *)D.out;
  __shared__ double smm[PMAX + 1], rdf[PMAX + 1];
  __shared__ double fa[KHALF_MAX], fb[KHALF_MAX];  // prefactor A(o, i) = fa[o] fb[i]
  __shared__ float faf[KHALF_MAX], fbf[KHALF_MAX];  // the same in FP32 (FP32 operators, p <= 12)
  bool cuse[ASM_CC];
  bool any = false;
#pragma unroll
  for (int k = 0; k < ASM_CC; ++k) {
    const int cls = cls0 + k;
    cuse[k] = cls < NREACT_CLS && (!D.used || D.used[cls]);
    any |= cuse[k];
  }
  if (!any) return;
  for (int k = 0; k < ASM_CC; ++k) {
    if (!cuse[k]) continue;
    const double *S = D.stab + ((size_t)(cls0 + k - D.cls0) * D.ntypes + D.tau) * TS;
    for (int e = threadIdx.x; e < (2 * p + 1) * NT * 4; e += blockDim.x) {
      const int d = e / (NT * 4), x = e % (NT * 4), Kk = d + 1 + 2 * (x >> 2);
      if (Kk <= KT)
        Sf[k * AS + d * AR + x] = df_split(sfac[Kk * (KMAX_TAB + 1) + d] * S[stab_index(KT, Kk, d, x & 3)]);
    }
  }
  if (threadIdx.x == 0) {
    double sg = 1.0;
    smm[0] = 1.0;
    for (int m = 1; m <= p; ++m) { sg *= -sqrt((2.0 * m + 1.0) / (2.0 * m)); smm[m] = sg; }
    rdf[0] = 1.0;
    for (int n = 1; n <= p; ++n) rdf[n] = rdf[n - 1] / (2.0 * n + 1.0);  // 1/(2n+1)!!
  }
  __syncthreads();
  // fa[o] = smm(m) st^{n-m} / (2n+1)!!,  fb[i] = smm(mu) (-st)^{nu-mu} / ((2nu+1)!! 4 pi h)
  for (int e = threadIdx.x; e < K; e += blockDim.x) {
    int n, m;
    hdecode(e, n, m);
    const bool odd = (n - m) & 1;
    fa[e] = smm[m] * rdf[n] * (odd ? (double)D.st : 1.0);
    fb[e] = smm[m] * rdf[n] * (odd ? -(double)D.st : 1.0) * (0.25 / PI) / D.h;
    faf[e] = (float)fa[e];
    fbf[e] = (float)fb[e];
  }
  __syncthreads();
  // FP32 epilogue for FP32 operators while the prefactors stay well inside the FP32 range
  const bool f32_out = sizeof(T) == 4 && p <= 12;
  const int NS = p + 2;
  const size_t KK = (size_t)K * K;
  for (int e = threadIdx.x; e < K * K; e += blockDim.x) {
    const int o = e / K, i = e % K;
    int n, m, nu, mu;
    hdecode(o, n, m);
    hdecode(i, nu, mu);
    const int ij = 2 * ((n - m) & 1) + ((nu - mu) & 1);
    const int smax = (n - m + 1) / 2 + (nu - mu + 1) / 2;
    const float2 *cf = D.coef + (size_t)e * NS;
    const int dp = mu - m, dm = mu + m;  // |d| for +mu and -mu
    const int adp = dp < 0 ? -dp : dp;
    float2 ap[ASM_CC], am[ASM_CC];
#pragma unroll
    for (int k = 0; k < ASM_CC; ++k) ap[k] = am[k] = make_float2(0.f, 0.f);
    // the entry's coefficients, all loads in flight at once (smax <= p + 1 < PMAX + 2)
    float2 cv[PMAX + 2];
#pragma unroll
    for (int s = 0; s < PMAX + 2; ++s) cv[s] = s <= smax ? cf[s] : make_float2(0.f, 0.f);
#pragma unroll
    for (int s = 0; s < PMAX + 2; ++s) {
      const int Kk = 1 + m + mu + 2 * s;
      if (s > smax || Kk > KT) break;
      const float2 c = cv[s];
      const int ip = adp * AR + ((m < mu ? m : mu) + s) * 4 + ij, im = dm * AR + s * 4 + ij;
#pragma unroll
      for (int k = 0; k < ASM_CC; ++k) {
        df_fma(c, Sf[k * AS + ip], ap[k]);
        df_fma(c, Sf[k * AS + im], am[k]);
      }
    }
    // signs: (-1)^|d| for d = mu - m < 0 and for d = -mu - m < 0; (-1)^mu of the -mu term
    const bool fp = dp < 0 && (adp & 1), fm = ((dm > 0 && (dm & 1)) != ((mu & 1) != 0));
#pragma unroll
    for (int k = 0; k < ASM_CC; ++k) {
      if (!cuse[k]) continue;
      const float2 Xd = fp ? make_float2(-ap[k].x, -ap[k].y) : ap[k];
      const float2 Yd = fm ? make_float2(-am[k].x, -am[k].y) : am[k];
      T *dP = out + (size_t)(cls0 + k) * D.ntypes * 2 * KK + (size_t)D.tau * 2 * KK + (size_t)o * K + i;
      T *dQ = dP + KK;
      if (f32_out) {
        const float Af = faf[o] * fbf[i];
        if (mu == 0) {
          *dP = (T)(Af * df_sum_f(Xd, make_float2(0.f, 0.f)));
          *dQ = (T)0;
        } else {
          *dP = (T)(Af * df_sum_f(Xd, Yd));
          *dQ = (T)(Af * df_sum_f(Xd, make_float2(-Yd.x, -Yd.y)));
        }
      } else {
        const double A = fa[o] * fb[i];
        const double X = (double)Xd.x + (double)Xd.y, Y = (double)Yd.x + (double)Yd.y;
        *dP = (T)(mu == 0 ? A * X : A * (X + Y));
        *dQ = (T)(mu == 0 ? 0.0 : A * (X - Y));
      }
    }
  }
}
static size_t assemble_smem(int p, int KT) { return ASM_CC * sizeof(float2) * (size_t)asm_size(p, KT); }

// near-field reaction quadrature nodes: W = w lr sigma / (4 pi lz_l), lz_l, lz_l'
__global__ void k_near_nodes(Medium md, int l, int a, int ntypes, double umax, double wmax, double lmin,
                             double *nodes, int nq) {
  __shared__ double pu[MAXPANEL], pw[MAXPANEL];
  __shared__ double gx[16], gw[16];
  __shared__ int npan;
  if (threadIdx.x == 0) {
    gl16(gx, gw);
    make_panels(umax, wmax, lmin, 0.5, pu, pw, &npan);
  }
  __syncthreads();
  const int tau = blockIdx.y;
  int lp, b;
  type_decode(tau, lp, b);
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < nq; j += gridDim.x * blockDim.x) {
    double *o = nodes + ((size_t)tau * nq + j) * 4;
    if (j >= npan * 16) { o[0] = o[1] = 0.0; o[2] = o[3] = 1.0; continue; }
    const int pi_ = j >> 4, gi = 15 - (j & 15);  // ascending abscissae
    const double lr = pu[pi_] + 0.5 * pw[pi_] * (gx[gi] + 1.0);
    const double w = 0.5 * pw[pi_] * gw[gi];
    const double lz = sqrt(md.lam[l] * md.lam[l] + lr * lr), lzp = sqrt(md.lam[lp] * md.lam[lp] + lr * lr);
    o[0] = lr;
    o[1] = w * lr * layer_sigma(md, lr, l, a, lp, b) / (4.0 * PI * lz);
    o[2] = lz;
    o[3] = lzp;
  }
}

// nodes, then tables, of nd descriptors
static void launch_nodes(Ctx &c, const RDesc *dr, const NDesc *dn, int nq, unsigned nd) {
  k_stab_nodes<<<dim3((unsigned)((nq + 127) / 128), nd), 128, 0, c.stream>>>(dr, dn, c.md);
  LPB_LAUNCH();
}
static void launch_tables(Ctx &c, const RDesc *dr, const NDesc *dn, unsigned nd, int KT) {
  LPB_ATTR_ONCE(k_stab_table, stab_table_smem(KMAX_TAB));  // the largest table any order needs
  k_stab_table<<<dim3(NKK * (NRHO / ST_NC), nd), ST_THREADS, stab_table_smem(KT), c.stream>>>(dr, dn, KT, c.sfac);
  LPB_LAUNCH();
}

// the free-space operators of every group: one launch of the radial factors, one of the operators
template <typename T>
static void build_free_t(Ctx &c, std::vector<Group> &groups) {
  const int p = c.p, K = c.K;
  const size_t KK = (size_t)K * K;
  std::vector<OpDesc> descs;
  size_t total = 0;
  auto add = [&](int kind, int out_inv, int in_inv, double lam, double bx, double by, double bz, double xout,
                 double xin, double pref, int dir, size_t offset_in_slot) {
    OpDesc d;
    d.kind = kind; d.out_inv = out_inv; d.in_inv = in_inv; d.dir = dir;
    d.lam = lam;
    d.bnorm = sqrt(bx * bx + by * by + bz * bz);
    d.cosb = bz / d.bnorm;
    d.xout = xout; d.xin = xin; d.pref = pref;
    d.dst = (int64_t)(total + offset_in_slot);
    descs.push_back(d);
  };
  // layout: per group and level a block with M2M (free + types), L2L, free M2L classes
  struct Blk { size_t m2m_t, m2m_i, l2l, fm2l; };
  std::vector<Blk> blk(groups.size() * (DMAX + 1));
  for (size_t gi = 0; gi < groups.size(); ++gi) {
    const Group &g = groups[gi];
    const int parts = g.parts;
    const double lam_t = c.md.lam[g.l];
    for (int l = 2; l <= g.D; ++l) {
      const double h = g.h(l), hc = h, hp = 2.0 * h;
      Blk b{};
      // M2M: children at level l -> parents at l-1 (only l >= 3)
      const bool free_l = g.is_free && (parts & 1) && l <= g.Df;  // free-space part lives at levels <= Df
      if (l >= 3) {
        if (free_l) {
          b.m2m_t = total;
          for (int cz = 0; cz < 2; ++cz)
            add(1, 1, 0, lam_t, 0.5 * hc, 0.5 * hc, (cz ? 0.5 : -0.5) * hc, lam_t * hp, lam_t * hc, 1.0,
                NFREE_CLS + cz, (size_t)cz * 2 * KK);
          total += 4 * KK;
        }
        if (parts & 2) {
          b.m2m_i = total;
          for (int t = 0; t < g.ntypes; ++t) {
            int lp, bb;
            type_decode(t, lp, bb);
            const double la = c.md.lam[lp];
            for (int cz = 0; cz < 2; ++cz)
              add(1, 1, 0, la, 0.5 * hc, 0.5 * hc, (cz ? 0.5 : -0.5) * hc, la * hp, la * hc, 1.0, NFREE_CLS + cz,
                  ((size_t)t * 2 + cz) * 2 * KK);
          }
          total += (size_t)g.ntypes * 4 * KK;
        }
        // L2L: parent (l-1) -> child at l
        b.l2l = total;
        for (int cz = 0; cz < 2; ++cz)
          add(2, 0, 1, lam_t, 0.5 * hc, 0.5 * hc, (cz ? 0.5 : -0.5) * hc, lam_t * hc, lam_t * hp, 1.0,
              NFREE_CLS + cz, (size_t)cz * 2 * KK);
        total += 4 * KK;
      }
      if (free_l) {
        b.fm2l = total;
        const double pref = lam_t / (2.0 * PI * PI * c.md.eps[g.l]);
        for (int ri = 0; ri < NRHO; ++ri)
          for (int dz = -OFF_R; dz <= OFF_R; ++dz) {
            const int cls = ri * NDZ + dz + OFF_R;
            if (!free_class_is_far(ri, dz, c.ws)) continue;
            // b = c_t - c_s = -(offset) h; azimuth factored out: b = (rho h, 0, -dz h)
            add(0, 0, 0, lam_t, sqrt((double)rho2_of(ri)) * h, 0.0, -dz * h, lam_t * h, lam_t * h, pref, cls,
                (size_t)cls * 2 * KK);
          }
        total += (size_t)NFREE_CLS * 2 * KK;
      }
      blk[gi * (DMAX + 1) + l] = b;
    }
  }
  T *ops = c.arena.get<T>(total);
  for (size_t gi = 0; gi < groups.size(); ++gi) {
    Group &g = groups[gi];
    for (int l = 2; l <= g.D; ++l) {
      const Blk &b = blk[gi * (DMAX + 1) + l];
      const bool free_l = g.is_free && (g.parts & 1) && l <= g.Df;
      g.op_m2m_t[l] = (l >= 3 && free_l) ? (void *)(ops + b.m2m_t) : nullptr;
      g.op_m2m_i[l] = (l >= 3 && (g.parts & 2)) ? (void *)(ops + b.m2m_i) : nullptr;
      g.op_l2l[l] = (l >= 3) ? (void *)(ops + b.l2l) : nullptr;
      g.op_free[l] = free_l ? (void *)(ops + b.fm2l) : nullptr;
    }
  }
  if (descs.empty()) return;
  OpDesc *dd = c.arena.get<OpDesc>(descs.size());
  LPB_CUDA(cudaMemcpyAsync(dd, descs.data(), sizeof(OpDesc) * descs.size(), cudaMemcpyHostToDevice, c.stream));
  double *prep = c.arena.get<double>(descs.size() * NPREP);
  k_ops_prep<<<(unsigned)((descs.size() + 63) / 64), 64, 0, c.stream>>>(dd, (int)descs.size(), p, prep);
  LPB_LAUNCH();
  k_build_ops<T><<<dim3((unsigned)descs.size(), OPS_SPLIT), 256, 0, c.stream>>>(dd, prep, c.phat_dir, p, K,
                                                                                c.gaunt, ops);
  LPB_LAUNCH();
  c.launches += 2;
}

// What the reaction tables and operators need of depths and medium alone: quadrature nodes, Bessel columns and
// Legendre-product coefficients of every group, level and type (three launches).  They run beside the trees and
// lists; in line with the tables, and those behind the free-space operators on one stream, they held up each
// small evaluation (N = 3,000, p = 10: 3.50 -> 3.31 ms with k_react_coef's and the assembly's shorter sums).
template <typename T>
static void begin_react_t(Ctx &c, std::vector<Group> &groups, ReactPlan &plan) {
  const int p = c.p, K = c.K;
  const size_t KK = (size_t)K * K;
  const int KT = 2 * p + 3, NS = p + 2;
  const size_t TS = (size_t)(KT + 1) * (KT + 1) * 4;
  std::vector<RDesc> &rd = plan.desc;
  for (auto &g : groups) {
    if (!(g.parts & 2) || !g.I.np || !g.T.np) continue;
    const int st = (g.a == 1) ? -1 : 1;
    for (int l = 2; l <= g.D; ++l) {
      const double h = g.h(l);
      g.stab[l] = c.arena.get<double>((size_t)NREACT_CLS * g.ntypes * TS);
      g.op_react[l] = c.arena.get<T>((size_t)NREACT_CLS * g.ntypes * 2 * KK);
      float2 *coef = c.arena.get<float2>((size_t)g.ntypes * KK * NS);
      for (int t = 0; t < g.ntypes; ++t) {
        int lp, bb;
        type_decode(t, lp, bb);
        RDesc d;
        d.l = g.l; d.a = g.a; d.lp = lp; d.b = bb; d.tau = t; d.ntypes = g.ntypes; d.st = st; d.lev = l;
        d.cls0 = 0; d.group = (int)(&g - groups.data());
        d.h = h; d.Lam = c.md.lam[g.l] * h; d.Lamp = c.md.lam[lp] * h;
        d.used = nullptr;
        d.stab = g.stab[l];
        d.coef = coef + (size_t)t * KK * NS;
        d.out = g.op_react[l];
        rd.push_back(d);
      }
    }
  }
  if (rd.empty()) return;
  RDesc *dr = c.arena.get<RDesc>(rd.size());
  LPB_CUDA(cudaMemcpyAsync(dr, rd.data(), sizeof(RDesc) * rd.size(), cudaMemcpyHostToDevice, c.stream));
  const unsigned nd = (unsigned)rd.size();
  // one node set for the whole evaluation (graded to the smallest Lambda of all reaction
  // groups), so the Bessel columns are evaluated once and shared
  NDesc N = node_desc(KT, fmax(c.tol, 1e-16), c.stab_lmin, c.stab_lmin);
  double *bes = c.arena.get<double>((size_t)N.nq * NBES);
  k_stab_bessel<<<(unsigned)(((int64_t)N.nq * NRHO + 255) / 256), 256, 0, c.stream>>>(N, bes);
  LPB_LAUNCH();
  N.bes = bes;
  std::vector<NDesc> nv(nd, N);
  for (auto &n : nv) n.nodes = c.arena.get<double>((size_t)N.nq * NDF);
  NDesc *dn = c.arena.get<NDesc>(nv.size());
  LPB_CUDA(cudaMemcpyAsync(dn, nv.data(), sizeof(NDesc) * nv.size(), cudaMemcpyHostToDevice, c.stream));
  plan.nodes = dn;
  launch_nodes(c, dr, dn, N.nq, nd);
  k_react_coef<<<dim3((unsigned)((KK + 255) / 256), nd), 256, sizeof(double) * 2 * K * c.tpk, c.stream>>>(
      dr, c.tpoly, c.tpk, p, K);
  LPB_LAUNCH();
  c.launches += 3;
}
// the tables and operators of the classes that the lists use (two launches)
template <typename T>
static void build_react_t(Ctx &c, std::vector<Group> &groups, ReactPlan &plan) {
  if (plan.desc.empty()) return;
  const int p = c.p, KT = 2 * p + 3;
  for (auto &d : plan.desc) d.used = groups[d.group].used[d.lev];
  const unsigned nd = (unsigned)plan.desc.size();
  RDesc *dr = c.arena.get<RDesc>(nd);
  LPB_CUDA(cudaMemcpyAsync(dr, plan.desc.data(), sizeof(RDesc) * nd, cudaMemcpyHostToDevice, c.stream));
  launch_tables(c, dr, plan.nodes, nd, KT);
  LPB_ATTR_ONCE(k_react_assemble<T>, assemble_smem(PMAX, KMAX_TAB));
  k_react_assemble<T><<<dim3((NREACT_CLS + ASM_CC - 1) / ASM_CC, nd), 256, assemble_smem(p, KT), c.stream>>>(
      dr, p, c.K, KT, c.sfac);
  LPB_LAUNCH();
  c.launches += 2;
}

void build_free_operators(Ctx &c, std::vector<Group> &groups) {
  c.opts.precision == LPBFMM_FP64 ? build_free_t<double>(c, groups) : build_free_t<float>(c, groups);
}
void begin_react_operators(Ctx &c, std::vector<Group> &groups, ReactPlan &plan) {
  c.opts.precision == LPBFMM_FP64 ? begin_react_t<double>(c, groups, plan) : begin_react_t<float>(c, groups, plan);
}
void build_react_operators(Ctx &c, std::vector<Group> &groups, ReactPlan &plan) {
  c.opts.precision == LPBFMM_FP64 ? build_react_t<double>(c, groups, plan) : build_react_t<float>(c, groups, plan);
}

void build_near_nodes(Ctx &c, Group &g, double zeta_min, double rho_max) {
  const double lmin = fmin(c.md.lam[g.l], [&] {
    double m = 1e300;
    for (int k = 0; k <= c.md.L; ++k) m = fmin(m, c.md.lam[k]);
    return m;
  }());
  const double umax = 36.0 / zeta_min;
  const double wmax = fmin(2.0 / zeta_min, PI / fmax(rho_max, 1e-300));
  g.nq = count_panels(umax, wmax, lmin, 0.5) * 16;
  g.nodes = c.arena.get<double>((size_t)g.ntypes * g.nq * 4);
  k_near_nodes<<<dim3((unsigned)((g.nq + 255) / 256), g.ntypes), 256, 0, c.stream>>>(c.md, g.l, g.a, g.ntypes, umax,
                                                                                     wmax, lmin, g.nodes, g.nq);
  LPB_LAUNCH();
  c.launches++;
}

// reaction class of a single-class table request: rho / h, zt / h - 1/2 and zs / h - 1/2 must be a
// class of the tables (rho^2 / h^2 one of the NRHO values, k_t + k_s < NKT)
static int class_of_request(double h, double rho, double zt, double zs) {
  const double r2 = (rho / h) * (rho / h);
  int ri = -1;
  for (int k = 0; k < NRHO; ++k)
    if (fabs(r2 - rho2_of(k)) < 1e-9) ri = k;
  const int kt = (int)llround(zt / h - 0.5), ks = (int)llround(zs / h - 0.5);
  const int kk = kk_index(kt, ks);
  if (ri < 0 || kk < 0 || fabs(zt / h - 0.5 - kt) > 1e-9 || fabs(zs / h - 0.5 - ks) > 1e-9)
    throw StatusError{LPBFMM_ERR_ARG};
  return ri * NKK + kk;
}

static RDesc one_class_desc(Ctx &c, int l, int a, int lp, int b, double h, int cls) {
  RDesc d;
  d.l = l; d.a = a; d.lp = lp; d.b = b; d.tau = 0; d.ntypes = 1; d.st = a == 1 ? -1 : 1; d.lev = 0;
  d.cls0 = cls; d.group = 0;
  d.h = h; d.Lam = c.md.lam[l] * h; d.Lamp = c.md.lam[lp] * h;
  d.used = nullptr; d.stab = nullptr; d.coef = nullptr; d.out = nullptr;
  return d;
}

void debug_stable(Ctx &c, int l, int a, int lp, int b, double h, double rho, double zt, double zs, int Kmax,
                  double *out) {
  // single class with the requested geometry: the quadrature + recurrence kernels of the FMM run
  // on a one-class descriptor whose table array holds that class alone
  const int cls = class_of_request(h, rho, zt, zs);
  const int KT = Kmax;
  const size_t TS = (size_t)(KT + 1) * (KT + 1) * 4;
  double *stab = nullptr;
  uint8_t *used = nullptr;
  RDesc *dr = nullptr;
  LPB_CUDA(cudaMalloc(&stab, sizeof(double) * TS));
  LPB_CUDA(cudaMalloc(&used, NREACT_CLS));
  LPB_CUDA(cudaMalloc(&dr, sizeof(RDesc)));
  LPB_CUDA(cudaMemsetAsync(stab, 0, sizeof(double) * TS, c.stream));
  std::vector<uint8_t> hu(NREACT_CLS, 0);
  hu[cls] = 1;
  LPB_CUDA(cudaMemcpyAsync(used, hu.data(), NREACT_CLS, cudaMemcpyHostToDevice, c.stream));
  RDesc d = one_class_desc(c, l, a, lp, b, h, cls);
  d.used = used;
  d.stab = stab;
  LPB_CUDA(cudaMemcpyAsync(dr, &d, sizeof(RDesc), cudaMemcpyHostToDevice, c.stream));
  const double tol = fmax(c.tol, 1e-16);
  NDesc N = node_desc(KT, tol, d.Lam, d.Lamp);
  NDesc *dn = nullptr;
  double *bes = nullptr;
  LPB_CUDA(cudaMalloc(&N.nodes, sizeof(double) * (size_t)N.nq * NDF));
  LPB_CUDA(cudaMalloc(&bes, sizeof(double) * (size_t)N.nq * NBES));
  LPB_CUDA(cudaMalloc(&dn, sizeof(NDesc)));
  k_stab_bessel<<<(unsigned)((N.nq * NRHO + 255) / 256), 256, 0, c.stream>>>(N, bes);
  LPB_LAUNCH();
  N.bes = bes;
  LPB_CUDA(cudaMemcpyAsync(dn, &N, sizeof(NDesc), cudaMemcpyHostToDevice, c.stream));
  launch_nodes(c, dr, dn, N.nq, 1);
  launch_tables(c, dr, dn, 1, KT);
  std::vector<double> h_out(TS);
  LPB_CUDA(cudaMemcpyAsync(h_out.data(), stab, sizeof(double) * TS, cudaMemcpyDeviceToHost, c.stream));
  LPB_CUDA(cudaStreamSynchronize(c.stream));
  cudaFree(stab);
  cudaFree(used);
  cudaFree(dr);
  cudaFree(N.nodes);
  cudaFree(bes);
  cudaFree(dn);
  // out[((K*(Kmax+1)) + d)*4 + ij] with ij = 2i + j
  for (size_t e = 0; e < TS; ++e) out[e] = h_out[e];
}


// ---------------------------------------------------------------------------------------
// Sommerfeld table of one class without any allocation.  Callers that cannot allocate: a
// host loop that has handed all free device memory to its own pool (cudaMalloc would fail),
// or one sharing the device with latency-critical streams (cudaMalloc and cudaFree may
// synchronize the whole device).  Every temporary lives in one fixed device array; its
// address is resolved per device with cudaGetSymbolAddress on the first call on that device.
// ---------------------------------------------------------------------------------------
constexpr size_t NA_TS = (size_t)(LPBFMM_NOALLOC_KMAX + 1) * (LPBFMM_NOALLOC_KMAX + 1) * 4;  // one class
constexpr size_t NA_NODES = (size_t)LPBFMM_NOALLOC_NQ * (NDF + NBES);  // doubles
constexpr size_t NA_DESC = (sizeof(RDesc) + sizeof(NDesc) + NREACT_CLS + 7) / 8 + 8;
constexpr size_t NA_DOUBLES = NA_TS + NA_NODES + NA_DESC;           // ~1.8 MB in all
static __device__ __align__(256) double g_noalloc_scratch[NA_DOUBLES];

static std::mutex g_noalloc_mu;
static double *g_noalloc_addr[LPB_MAX_DEVICES] = {};

// the scratch array's device address on the context's device (which must be current)
static double *noalloc_scratch(const Ctx &c) {
  int dev = -1;
  LPB_CUDA(cudaGetDevice(&dev));
  if (dev != c.device) throw StatusError{LPBFMM_ERR_ARG};
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (!g_noalloc_addr[c.device]) {
    void *p = nullptr;
    LPB_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch));
    g_noalloc_addr[c.device] = (double *)p;
  }
  return g_noalloc_addr[c.device];
}

// descriptors, class mask and the class's table are (re)initialised by one launch: the table
// entries the kernels do not write (d > K, and d >= 2 with K < d + 1) must read as zero
__global__ void k_noalloc_init(RDesc d, NDesc n, RDesc *rd, NDesc *nd, uint8_t *used, int cls, double *stab_cls,
                               int ts) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  if (t == 0) {
    *rd = d;
    *nd = n;
  }
  for (int e = t; e < NREACT_CLS; e += stride) used[e] = (e == cls) ? 1 : 0;
  for (int e = t; e < ts; e += stride) stab_cls[e] = 0.0;
}

void stable_noalloc(Ctx &c, int l, int a, int lp, int b, double h, double rho, double zt, double zs, int Kmax,
                    double *out) {
  if (Kmax > LPBFMM_NOALLOC_KMAX) throw StatusError{LPBFMM_ERR_UNSUPPORTED};
  const int cls = class_of_request(h, rho, zt, zs);
  const int KT = Kmax;
  const size_t TS = (size_t)(KT + 1) * (KT + 1) * 4;
  RDesc d = one_class_desc(c, l, a, lp, b, h, cls);
  NDesc N = node_desc(KT, fmax(c.tol, 1e-16), d.Lam, d.Lamp);
  // the limit counts 16-point panels of width 2, the rule it was set for; the present rule needs fewer nodes
  if (count_panels(N.umax, 2.0, N.lmin, 0.5) * 16 > LPBFMM_NOALLOC_NQ || N.nq > LPBFMM_NOALLOC_NQ)
    throw StatusError{LPBFMM_ERR_UNSUPPORTED};
  double *base = noalloc_scratch(c);
  double *stab = base, *nodes = base + NA_TS;
  RDesc *dr = (RDesc *)(nodes + NA_NODES);
  NDesc *dn = (NDesc *)((char *)dr + ((sizeof(RDesc) + 15) / 16) * 16);
  uint8_t *used = (uint8_t *)((char *)dn + ((sizeof(NDesc) + 15) / 16) * 16);
  d.used = used;
  d.stab = stab;
  N.nodes = nodes;
  double *bes = nodes + (size_t)LPBFMM_NOALLOC_NQ * NDF;
  k_stab_bessel<<<(unsigned)((N.nq * NRHO + 255) / 256), 256, 0, c.stream>>>(N, bes);
  LPB_LAUNCH();
  N.bes = bes;
  k_noalloc_init<<<8, 256, 0, c.stream>>>(d, N, dr, dn, used, cls, stab, (int)TS);
  LPB_LAUNCH();
  launch_nodes(c, dr, dn, N.nq, 1);
  launch_tables(c, dr, dn, 1, KT);
  LPB_CUDA(cudaMemcpyAsync(out, stab, sizeof(double) * TS, cudaMemcpyDeviceToDevice, c.stream));
}

}  // namespace lpb
