// Host engine of librs: contexts, prepared batches, CUDA-graph replay and the
// C ABI of include/rs.h.  The host plans (planner.cpp), packs inputs into one
// pinned staging buffer, enqueues G1 (kernels_g1.cu), G2 and G3
// (kernels_g23.cu) on a stream and unpacks the results.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <thread>

#include "engine.h"

namespace {

thread_local std::string g_err;

constexpr size_t kAlign = 256;
size_t align_up(size_t x) { return (x + kAlign - 1) & ~(kAlign - 1); }

// Whether G1 evaluates plan p (register capacity C) through its threads'
// columns of shared memory: unless they leave an SM room for one block of 128
// threads (or none, at C = 72) where the staged coefficients alone leave room
// for two.  G1, ns per image, degrees in x and y of f and g; before there were
// columns, with them, without:
//   (300, 71) (1, 8)    1 and 2 blocks    3.61   4.36   3.14
//   (400, 55) (1, 12)   1 and 2           3.10   3.88   2.63
//   (660, 71) (1, 4)    none and 1        8.99   14.5 (64 threads)   8.03
//   (200, 38) (200, 38) 2 and 3           2.15   1.97   1.94
//   (250, 30) (250, 30) 2 and 3           1.99   1.81   1.71
//   (150, 44) (150, 44) 2 and 3           2.24   2.12   2.19
//   (150, 38) (150, 38) 3 and 4           1.81   1.49   1.54
//   (100, 70) (100, 70) 2 and 2           3.76   3.03   3.32
//   (500, 71) (1, 8)    1 and 1           6.85   5.70   6.09
static bool rs_g1_column(const PairPlan &p, int C) {
  auto blocks = [&](bool col) { return (227 * 1024) / (rs_g1_smem_words(p, C, 128, col) * 4 + 1024); };
  return blocks(true) > 1 || blocks(true) == blocks(false);
}

// Modular products of the normal remainder sequence (a4 count): three per
// coefficient of a double step, two of the single step between equal degrees.
double prs_products(int a, int b) {
  double u = 0;
  while (a > 0 && b > 0) {
    if (a == b) {
      u += 2.0 * a;
      --a;
    } else if (a > b) {
      u += 3.0 * (a - 1);
      a -= 2;
    } else {
      u += 3.0 * (b - 1);
      b -= 2;
    }
  }
  return u;
}

}  // namespace

int rs_cuda_code(cudaError_t e) { return e == cudaErrorMemoryAllocation ? RS_ERR_NOMEM : RS_ERR_CUDA; }

int rs_fail(rs_ctx *c, int code, const std::string &msg) {
  if (c)
    c->err = msg;
  else
    g_err = msg;
  return code;
}

#define RS_CUDA(ctx, call)                                                                         \
  do {                                                                                             \
    cudaError_t e_ = (call);                                                                       \
    if (e_ != cudaSuccess)                                                                         \
      return rs_fail((ctx), rs_cuda_code(e_), std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

// ------------------------------------------------------------------ planning

// Host threads for planning n pairs, and pairs per task.  Planning reads every
// input coefficient once and takes one summed autocorrelation per polynomial
// ((deg_x + 1)^2 (deg_y + 1) / 2 products); on the Grace host it takes about
// 0.6 us per polynomial, 5 ns per coefficient and 1 ns per limb, and 0.5 ns
// per product.  From 60 us on the pairs are shared: a worker takes a few
// microseconds to wake.
static int plan_threads(int n, const rs_bipoly *f, const rs_bipoly *g, int *step) {
  auto cost = [](const rs_bipoly &p) {  // ns
    if (!p.coeffs || p.deg_x < 0 || p.deg_y < 0 || p.limbs < 1 || p.limbs > RS_MAX_LIMBS) return 0.0;
    const double c = ((double)p.deg_x + 1) * ((double)p.deg_y + 1);
    return 600.0 + c * (5.0 + p.limbs) + (c <= 0x1p26 ? 0.25 * c * (p.deg_x + 1) : 0.0);
  };
  double ns = 0.0;
  for (int i = 0; i < n; ++i) ns += cost(f[i]) + cost(g[i]);
  const int threads = ns < 60e3 ? 1 : (int)std::min(16.0, ns / 20e3);
  *step = std::max(1, n / (8 * threads));
  return threads;
}

static void plan_one(rs_ctx *ctx, const rs_bipoly &f, const rs_bipoly &g, PairPlan &plan, const char **why) {
  try {
    plan.status = rs_plan_pair(&f, &g, ctx->log2p, plan, why);
  } catch (const std::exception &) {
    plan.status = RS_ERR_NOMEM;
    *why = "out of host memory";
  }
}

int rs_plan_all(rs_ctx *ctx, int n, const rs_bipoly *f, const rs_bipoly *g,
                std::vector<PairPlan> &plans, int32_t *status, int *first_err) {
  plans.assign(n, PairPlan());
  *first_err = RS_OK;
  std::vector<const char *> why(n, "");
  int step = 1;
  const int threads = plan_threads(n, f, g, &step);
  ctx->pool.run((n + step - 1) / step, threads, [&](int t) {
    for (int i = t * step; i < std::min(n, (t + 1) * step); ++i) plan_one(ctx, f[i], g[i], plans[i], &why[i]);
  });
  for (int i = 0; i < n; ++i) {
    const int rc = plans[i].status;
    if (status) status[i] = rc;
    if (rc != RS_OK && *first_err == RS_OK) {
      *first_err = rc;
      rs_fail(ctx, rc, std::string("pair ") + std::to_string(i) + ": " + why[i]);
    }
  }
  return *first_err;
}

bool rs_same_shape(const PairPlan &a, const PairPlan &b) {
  return a.status == b.status && a.trivial_zero == b.trivial_zero && a.N == b.N && a.K == b.K &&
         a.Kcrt == b.Kcrt &&
         a.Lout == b.Lout && a.f.my == b.f.my && a.g.my == b.g.my && a.f.mx == b.f.mx &&
         a.g.mx == b.g.mx && a.f.L == b.f.L && a.g.L == b.g.L && a.f.stride == b.f.stride &&
         a.g.stride == b.g.stride && a.f.dx == b.f.dx && a.g.dx == b.g.dx;
}

int64_t rs_input_words(const rs_bipoly &p) { return (int64_t)(p.deg_x + 1) * (p.deg_y + 1) * p.limbs; }

// ------------------------------------------------------------------ tables

static void free_tables(RsTables &t) {
  void *p[] = {t.finv, t.gtab, t.qn, t.btab, t.qc, t.qp, t.hq, t.wtab, t.wtri, t.p16, t.poff, t.nh};
  for (void *x : p)
    if (x) cudaFree(x);
  t = RsTables();
}

// Reserved 16-bit digits of row k of the prefix-product table: p_0 ... p_{k-1}
// < 2^(31 k), rounded up to a multiple of 32.
static int p16_row(int k) { return ((31 * k) / 16 + 2 + 31) / 32 * 32; }

// ------------------------------------------------------------ NTT tables

// The three NTT primes c 2^k + 1 (k >= 25) of the transform-based G2, in
// (2^30, 2^31) and ascending; their product exceeds 2^92.
static const uint32_t kNttPrimes[3] = {1811939329u, 2013265921u, 2113929217u};

static uint32_t powmod_u32(uint64_t a, uint64_t e, uint32_t P) {
  uint64_t r = 1;
  a %= P;
  while (e) {
    if (e & 1) r = r * a % P;
    a = a * a % P;
    e >>= 1;
  }
  return (uint32_t)r;
}

// Smallest generator of Z_P^* (P prime): g^((P-1)/r) != 1 for every prime r | P - 1.
static uint32_t generator_of(uint32_t P) {
  std::vector<uint32_t> fac;
  uint32_t n = P - 1;
  for (uint32_t r = 2; (uint64_t)r * r <= n; ++r)
    if (n % r == 0) {
      fac.push_back(r);
      while (n % r == 0) n /= r;
    }
  if (n > 1) fac.push_back(n);
  for (uint32_t g = 2;; ++g) {
    bool ok = true;
    for (uint32_t r : fac) ok = ok && powmod_u32(g, (P - 1) / r, P) != 1;
    if (ok) return g;
  }
}

// Constants and twiddles [q][forward, inverse][2^LGMAX] as (w, floor(w 2^32 / P)):
// for each length 2^lg a row of w_L^j (forward) or w_L^-j (inverse), j < 2^(lg-1),
// starting at 2^(lg-1) - 1.
static void ntt_host_tables(NttConst &nc, std::vector<uint2> &tw) {
  const int ROW = 1 << RS_NTT_LGMAX;
  tw.assign((size_t)6 * ROW, make_uint2(0, 0));
  for (int q = 0; q < 3; ++q) {
    const uint32_t P = kNttPrimes[q];
    nc.m[q] = make_modp(P);
    const uint32_t wmax = powmod_u32(generator_of(P), (P - 1) >> RS_NTT_LGMAX, P);
    for (int lg = 1; lg <= RS_NTT_LGMAX; ++lg) {
      const uint32_t w = powmod_u32(wmax, (uint64_t)1 << (RS_NTT_LGMAX - lg), P);
      const uint32_t wi = powmod_u32(w, P - 2, P);
      const int n = 1 << (lg - 1);
      uint64_t f = 1, b = 1;
      for (int j = 0; j < n; ++j) {
        tw[(size_t)(2 * q) * ROW + (n - 1) + j] = make_uint2((uint32_t)f, (uint32_t)((f << 32) / P));
        tw[(size_t)(2 * q + 1) * ROW + (n - 1) + j] = make_uint2((uint32_t)b, (uint32_t)((b << 32) / P));
        f = f * w % P;
        b = b * wi % P;
      }
    }
  }
  const uint32_t P0 = kNttPrimes[0], P1 = kNttPrimes[1], P2 = kNttPrimes[2];
  const uint64_t R1 = ((uint64_t)1 << 32) % P1, R2 = ((uint64_t)1 << 32) % P2;
  nc.c01 = (uint32_t)((uint64_t)powmod_u32(P0, P1 - 2, P1) * R1 % P1);
  nc.p0_m2 = (uint32_t)((uint64_t)P0 % P2 * R2 % P2);
  const uint32_t p01 = (uint32_t)((uint64_t)P0 * P1 % P2);
  nc.c012 = (uint32_t)((uint64_t)powmod_u32(p01, P2 - 2, P2) * R2 % P2);
}

int rs_g2_len(int N) {
  int lg = 1;
  while ((1 << lg) < 2 * N - 1) ++lg;
  return lg <= RS_NTT_LGMAX ? lg : 0;
}

// Cost per (pair, prime) of interpolating N point pairs, in units of 0.37 ps of
// the whole GPU.  Direct: one unit per N^2 (two multiply-accumulates) and 170
// per point for the rest of the kernel (12 ns at N = 113, 1.56 us at 2,049).
// Transforms: 12 of (L/2) lg radix-4 butterflies, 6.5 units each (1.60 us at
// N = 2,049, L = 2^13).
double rs_g2_cost(int N, int form) {
  const int lg = rs_g2_len(N);
  if (form == 0 || lg == 0) return (double)N * N + 170.0 * N;
  return 12.0 * 6.5 * (double)(1 << (lg - 1)) * lg + 60.0 * N;
}

// Launch shape of the direct form for M point pairs: the threads of a block,
// the segments of a block pair's walk, the halves (E, O) at once, and whether
// E and O get a block each (a cluster of two); see g2_kernel.  The least of an
// estimate in cycles of the busiest SM, fitted to sweeps over 32 to 512
// threads: a warp's step (one chunk, 56 wide products) takes 277 cycles of its
// scheduler, or 622 from start to end alone; the rest of a block 1,900 per warp
// and 550 per warp, half and round over the points, and 5,000 from start to
// end.  Measured (us, G2 stage): 40,000 tasks of M = 113: 427 with 32 threads
// (2 rounds, 3 segments), 474, 597, 986 and 1,599 with 64, 128, 256 and 512;
// 546 of 2,049: 1,140, 1,027, 984 and 853 with 64, 128, 256 and 512; 69 of 451:
// 20.2 with 384 threads in clusters, 24.2 with the best single blocks (all
// before the first loads were taken together, which changed no order here).
RsG2Shape rs_g2_shape(int M, int64_t tasks, int sms, const RsG2Shape *like) {
  static const int kT[8] = {32, 64, 96, 128, 192, 256, 384, 512};
  const int nblk = (M + RS_CONV_R - 1) / RS_CONV_R, npair = (nblk + 1) / 2, W = M + 2 * RS_G2_PAD;
  RsG2Shape best{256, 1, 1, 0, (size_t)(3 * W + M) * 4};
  double tbest = 1e300;
  for (int split = 0; split < 2; ++split) {
    if (like && split != like->split) continue;
    const int nh = split ? 1 : 2;
    const int64_t n = ((tasks << split) + sms - 1) / sms;  // blocks of the busiest SM
    if (split && n > 4 && !like) continue;
    for (int T : kT) {
      if (like && T != like->threads) continue;
      for (int rounds = 1; rounds <= 2; ++rounds) {
        const int S = std::max(1, std::min(std::min(nblk + 1, 16), rounds * T / (nh * npair)));
        const size_t smem = (size_t)((nh + 1) * W + S * nh * M) * 4;
        if (smem > (size_t)RS_G2_MAX_SMEM_BYTES) continue;
        const int len = (nblk + S) / S, units = nh * npair * S, iters = (M + T - 1) / T;
        const int64_t res = std::max<int64_t>(1, std::min<int64_t>(std::min(32, 1024 / T), (226 * 1024) / (smem + 1536)));
        const double rest = 550.0 * nh * iters;
        const double busy = n * 0.25 * (2.0 * len * ((units + 31) / 32) * 277.0 + T / 32 * (1900.0 + rest));
        const double path = ((n + res - 1) / res) * (2.0 * len * ((units + T - 1) / T) * 622.0 + 5000.0 + rest);
        const double t = busy * busy + 4.0 * path * path;
        if (t < tbest) {
          tbest = t;
          best = RsG2Shape{T, S, nh, split, smem};
        }
      }
    }
  }
  return best;
}

int rs_ensure_bhat(rs_ctx *ctx, int lg, int K) {
  const int L = 1 << lg;
  int rc = rs_ensure_tables(ctx, K, L / 2, 0);  // b_t for every t < L/2
  if (rc != RS_OK) return rc;
  std::lock_guard<std::mutex> lock(ctx->tab_mu);
  if (ctx->bhat_K[lg] >= K) return RS_OK;
  const RsTables &t = ctx->tab;
  DevGuard dg(ctx->device);
  uint32_t *nb = nullptr;
  cudaError_t e = cudaMalloc(&nb, (size_t)t.K * 3 * L * 4);
  if (e == cudaSuccess) e = launch_bhat(t.btab, t.N, t.N, t.K, lg, ctx->d_ntt_tw, ctx->nttc, nb, ctx->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  if (e != cudaSuccess) {
    if (nb) cudaFree(nb);
    return rs_fail(ctx, rs_cuda_code(e), std::string("transform tables: ") + cudaGetErrorString(e));
  }
  if (ctx->bhat[lg]) ctx->bhat_retired.push_back(ctx->bhat[lg]);
  ctx->bhat[lg] = nb;
  ctx->bhat_K[lg] = t.K;
  return RS_OK;
}

int rs_ensure_g2t_btile(rs_ctx *ctx, int K, int tiles) {
  std::lock_guard<std::mutex> lock(ctx->tab_mu);
  if (ctx->g2t_K >= K && ctx->g2t_tiles >= tiles) return RS_OK;
  const RsTables &t = ctx->tab;
  const int nK = std::max(K, ctx->g2t_K), nt = std::max(tiles, ctx->g2t_tiles);
  if (t.K < nK)
    return rs_fail(ctx, RS_ERR_STATE, "tensor-core G2 tables: point tables not built for these primes");
  DevGuard dg(ctx->device);
  uint16_t *nb = nullptr;
  cudaError_t e = cudaMalloc(&nb, (size_t)nK * nt * 8192 * sizeof(uint16_t));
  if (e == cudaSuccess) e = launch_g2t_btile(t.btab, t.N, t.N, nK, nt, nb, ctx->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  if (e != cudaSuccess) {
    if (nb) cudaFree(nb);
    return rs_fail(ctx, rs_cuda_code(e), std::string("tensor-core G2 tables: ") + cudaGetErrorString(e));
  }
  if (ctx->g2t_bt) ctx->g2t_retired.push_back(ctx->g2t_bt);
  ctx->g2t_bt = nb;
  ctx->g2t_K = nK;
  ctx->g2t_tiles = nt;
  return RS_OK;
}

int rs_ensure_g3m_wtiles(rs_ctx *ctx, int KB) {
  std::lock_guard<std::mutex> lock(ctx->tab_mu);
  if (ctx->g3m_KB >= KB) return RS_OK;
  const RsTables &t = ctx->tab;
  if (t.K < 64 * (KB - 1))
    return rs_fail(ctx, RS_ERR_STATE, "tensor-core CRT tables: CRT tables not built for these primes");
  DevGuard dg(ctx->device);
  uint16_t *nw = nullptr, *nr = nullptr;
  cudaError_t e = cudaMalloc(&nw, (size_t)std::max<int64_t>(1, g3m_wtile_elems(KB)) * sizeof(uint16_t));
  if (e == cudaSuccess) e = cudaMalloc(&nr, (size_t)std::max<int64_t>(1, g3m_rtile_elems(KB)) * sizeof(uint16_t));
  if (e == cudaSuccess) e = launch_g3m_wtiles(t.wtab, t.K, KB, nw, ctx->stream);
  if (e == cudaSuccess) e = launch_g3m_rtiles(t.wtab, t.K, KB, nr, ctx->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  if (e != cudaSuccess) {
    if (nw) cudaFree(nw);
    if (nr) cudaFree(nr);
    return rs_fail(ctx, rs_cuda_code(e), std::string("tensor-core CRT tables: ") + cudaGetErrorString(e));
  }
  if (ctx->g3m_wt) ctx->g3m_retired.push_back(ctx->g3m_wt);
  if (ctx->g3m_rt) ctx->g3m_retired.push_back(ctx->g3m_rt);
  ctx->g3m_wt = nw;
  ctx->g3m_rt = nr;
  ctx->g3m_KB = KB;
  return RS_OK;
}

// Chunk c's prefix products reach byte 2 nh[k] (balanced digits of P_k, k
// its last prime's row) and, shifted by up to three digits, column
// 2 nh[k] + 3: units 0 .. (2 nh[k] + 3) / 256 get a block each.
int rs_ensure_g3l_tiles(rs_ctx *ctx, int KB) {
  std::lock_guard<std::mutex> lock(ctx->tab_mu);
  if (ctx->g3l_KB >= KB) return RS_OK;
  const RsTables &t = ctx->tab;
  if (t.K < 64 * (KB - 1) || (int)t.h_nh.size() < t.K + 1)
    return rs_fail(ctx, RS_ERR_STATE, "tensor-core CRT limb tables: CRT tables not built for these primes");
  std::vector<int32_t> cbase(KB + 1, 0);
  for (int c = 0; c < KB; ++c) {
    const int klast = std::min(64 * c + 63, t.K);
    cbase[c + 1] = cbase[c] + (2 * t.h_nh[klast] + 3) / 256 + 1;
  }
  DevGuard dg(ctx->device);
  uint16_t *nw = nullptr;
  int32_t *ncb = nullptr;
  cudaError_t e = cudaMalloc(&nw, (size_t)cbase[KB] * g3l_block_elems() * sizeof(uint16_t));
  if (e == cudaSuccess) e = cudaMalloc(&ncb, cbase.size() * sizeof(int32_t));
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(ncb, cbase.data(), cbase.size() * sizeof(int32_t), cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess) e = launch_g3l_btiles(t.p16, t.poff, t.K, ncb, KB, cbase[KB], nw, ctx->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  if (e != cudaSuccess) {
    if (nw) cudaFree(nw);
    if (ncb) cudaFree(ncb);
    return rs_fail(ctx, rs_cuda_code(e), std::string("tensor-core CRT limb tables: ") + cudaGetErrorString(e));
  }
  if (ctx->g3l_bt) ctx->g3m_retired.push_back(ctx->g3l_bt);
  if (ctx->g3l_cbase) ctx->g3m_retired.push_back(ctx->g3l_cbase);
  ctx->g3l_bt = nw;
  ctx->g3l_cbase = ncb;
  ctx->h_g3l_cbase = cbase;
  ctx->g3l_KB = KB;
  return RS_OK;
}

int rs_ensure_tables(rs_ctx *ctx, int K, int N, int dx) {
  std::lock_guard<std::mutex> lock(ctx->tab_mu);
  const int need_c = N + 128 + dx + 1;
  RsTables &t = ctx->tab;
  if (K <= t.K && N <= t.N && need_c <= t.cstride) return RS_OK;
  RsTables nt;
  nt.K = std::min((int)ctx->primes.size(), ((std::max(K, t.K) + 63) / 64) * 64);
  nt.N = ((std::max(N, t.N) + 255) / 256) * 256;
  nt.cstride = ((std::max(need_c, t.cstride) + 255) / 256) * 256;
  DevGuard dg(ctx->device);
  const size_t ni = (size_t)nt.K * nt.N * 4, nc = (size_t)nt.K * nt.cstride * 4;
  cudaError_t e = cudaMalloc(&nt.finv, ni);
  if (e == cudaSuccess) e = cudaMalloc(&nt.gtab, ni);
  if (e == cudaSuccess) e = cudaMalloc(&nt.btab, ni);
  if (e == cudaSuccess) e = cudaMalloc(&nt.hq, ni);
  if (e == cudaSuccess) e = cudaMalloc(&nt.qc, nc);
  if (e == cudaSuccess) e = cudaMalloc(&nt.qn, nc);
  if (e == cudaSuccess) e = cudaMalloc(&nt.qp, nc);
  if (e == cudaSuccess)
    e = launch_tables(ctx->d_mods, ctx->d_qbase, nt.K, nt.N, nt.cstride, nt.finv, nt.gtab, nt.btab,
                      nt.hq, nt.qc, nt.qn, nt.qp, ctx->stream);
  // Chinese-remaindering tables for the same primes.
  // Rows 0..K of the prefix products: row K (the product of all K primes of
  // a pair that uses every table prime) gives floor(P / 2) to the limb kernel.
  std::vector<int32_t> poff(nt.K + 2, 0);
  for (int k = 0; k <= nt.K; ++k) poff[k + 1] = poff[k] + p16_row(k);
  if (e == cudaSuccess) e = cudaMalloc(&nt.wtab, std::max<size_t>(1, (size_t)nt.K * (nt.K - 1) / 2) * 4);
  if (e == cudaSuccess) e = cudaMalloc(&nt.wtri, (size_t)crt_tri_words(nt.K) * 4);
  if (e == cudaSuccess) e = cudaMalloc(&nt.p16, (size_t)poff[nt.K + 1] * 2);
  if (e == cudaSuccess) e = cudaMalloc(&nt.poff, (size_t)(nt.K + 2) * 4);
  if (e == cudaSuccess) e = cudaMalloc(&nt.nh, (size_t)(nt.K + 1) * 4);
  // Prefix products P_k = p_0 ... p_{k-1} as 16-bit digits (row k at poff[k],
  // zero padded to its reserved length; read as 32-bit limbs by the limb
  // kernels) and nh[k] = digits up to the top non-zero one, built on the
  // host: P_{k+1} = P_k p_k on 32-bit limbs.
  std::vector<uint16_t> p16((size_t)poff[nt.K + 1], 0);
  std::vector<int32_t> nh(nt.K + 1, 0);
  {
    std::vector<uint32_t> limbs(1, 1u);
    for (int k = 0; k <= nt.K; ++k) {
      uint16_t *row = p16.data() + poff[k];
      const int reserved = poff[k + 1] - poff[k];
      int top = 0;
      for (int i = 0; i < reserved && (i >> 1) < (int)limbs.size(); ++i) {
        const uint32_t d = (i & 1) ? (limbs[i >> 1] >> 16) : (limbs[i >> 1] & 0xffffu);
        row[i] = (uint16_t)d;
        if (d) top = i + 1;
      }
      nh[k] = top;
      if (k == nt.K) break;
      uint64_t carry = 0;
      for (uint32_t &l : limbs) {
        const uint64_t v = (uint64_t)l * ctx->primes[k] + carry;
        l = (uint32_t)v;
        carry = v >> 32;
      }
      if (carry) limbs.push_back((uint32_t)carry);
    }
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(nt.poff, poff.data(), poff.size() * 4, cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(nt.p16, p16.data(), p16.size() * 2, cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(nt.nh, nh.data(), nh.size() * 4, cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess) e = launch_crt_tables(ctx->d_mods, ctx->d_crt, nt.K, nt.wtab, nt.wtri, ctx->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  if (e != cudaSuccess) {
    free_tables(nt);
    return rs_fail(ctx, rs_cuda_code(e), std::string("point tables: ") + cudaGetErrorString(e));
  }
  nt.h_nh = nh;
  if (t.finv) ctx->retired.push_back(t);
  t = nt;
  return RS_OK;
}

// ------------------------------------------------------------------ batches

void rs_free_batch(rs_batch *b) {
  if (!b) return;
  DevGuard dg(b->ctx->device);
  if (b->gexec) cudaGraphExecDestroy(b->gexec);
  for (auto &e : b->ev)
    if (e) cudaEventDestroy(e);
  for (auto &e : b->fev)
    if (e) cudaEventDestroy(e);
  for (auto &e : b->jev)
    if (e) cudaEventDestroy(e);
  for (auto &e : b->cev) cudaEventDestroy(e);
  if (b->arena) {
    if (b->opt.stream_ordered)
      cudaFreeAsync(b->arena, b->stream);
    else
      cudaFree(b->arena);
  }
  if (b->own_host) {
    if (b->h_in) cudaFreeHost(b->h_in);
    if (b->h_out) cudaFreeHost(b->h_out);
  }
  delete b;
}

void rs_batch_sizes(const std::vector<PairPlan> &plans, int64_t *in_words, int64_t *out_words,
                    int64_t *device_bytes) {
  int64_t in = 0, out = 0, img = 0, meta = 0, tiles = 0, g2 = 0, g3 = 0, xl = 0, cy = 0, g3d = 0, g3b = 0;
  int64_t t_items = 0, t_bytes = 0;  // tensor-core G2 work items and buffers, if every pair takes that form
  for (size_t i = 0; i < plans.size(); ++i) {
    const PairPlan &p = plans[i];
    in += rs_used_words(p, p.f) + rs_used_words(p, p.g);
    if (p.status != RS_OK || p.trivial_zero) continue;
    const int64_t chunks = (p.Lout + 15) / 16;
    out += (int64_t)p.N * p.Lout + 2;
    xl += (int64_t)p.N * 16 * chunks;
    cy += (int64_t)p.N * chunks;
    img += (int64_t)p.K * 2 * ((p.N + 1) / 2);
    meta += p.f.my + p.g.my + 2;
    tiles += (int64_t)p.K * (((p.N + 1) / 2 + 15) / 16);
    g2 += p.K;
    const int64_t mt = (((p.N + 1) / 2 + 63) / 64) * 64;
    t_items += (int64_t)p.K * (mt / 64);
    t_bytes += (int64_t)p.K * mt * 2 * (4 * 2 + 4);  // two rows: four bf16 digits and one product per input
    t_bytes += (int64_t)((p.N + 127) / 128) * (((p.K + 63) / 64) * 65536 + 8);  // tensor-core CRT digit rows
    g3 += (p.N + 127) / 128;
    g3d += (p.N + 31) / 32;  // digit tiles
    g3b += (p.N + 127) / 128 * chunks;
  }
  // inputs plus room for the static tables (descriptors, tiles, task lists)
  // that rs_build_batch packs behind them in borrowed pinned staging
  const int64_t stat = meta * 2 + (int64_t)plans.size() * (int64_t)(sizeof(PairDesc) / 4) + tiles * 4 +
                       g2 * 2 + g3 * 2 + g3d * 4 + g3b * 4 + 8 * 4 + g2 * 4 + g2 * 8 + t_items * 2;
  *in_words = in + stat;
  *out_words = out + 1;
  *device_bytes = (int64_t)(align_up(in * 4) + align_up(meta * 8) + align_up(plans.size() * sizeof(PairDesc)) +
                            align_up(tiles * sizeof(Tile)) + kAlign + 2 * align_up(img * 4) +
                            align_up(xl * 4) + align_up(out * 4) + align_up(cy * 8) + align_up(g2 * 8) +
                            align_up(g3 * 8) + align_up(g3d * 8) + align_up(g3b * 16) + kAlign +
                            align_up(g2 * 16) + align_up(g2 * 32) + align_up(t_items * 8) + align_up(t_bytes));
}

int rs_build_batch(rs_ctx *ctx, int n, const rs_bipoly *f, const rs_bipoly *g,
                   std::vector<PairPlan> &&plans, const RsBatchOpts &opt, rs_batch **out) {
  rs_batch *b = new rs_batch();
  b->ctx = ctx;
  b->n = n;
  b->opt = opt;
  b->stream = opt.stream ? opt.stream : ctx->stream;
  b->plans = std::move(plans);
  b->dev_index.assign(n, -1);
  memset(&b->info, 0, sizeof(b->info));
  b->info.pairs = n;
  const bool images_only = opt.images_only;

  std::vector<int2> meta;
  std::vector<int> order;
  b->in_f.assign(n, -1);
  b->in_g.assign(n, -1);
  int maxM = 1, maxK = 0, maxDx = 0;  // largest point-pair count, prime count, x-degree
  for (int i = 0; i < n; ++i) {
    const PairPlan &p = b->plans[i];
    b->in_f[i] = b->in_words;
    b->in_words += rs_used_words(p, p.f);
    b->in_g[i] = b->in_words;
    b->in_words += rs_used_words(p, p.g);
    if (p.status != RS_OK || p.trivial_zero) continue;
    PairDesc d;
    memset(&d, 0, sizeof(d));
    d.my = p.f.my;
    d.ny = p.g.my;
    d.N = p.N;
    d.NI = 2 * ((p.N + 1) / 2);
    d.K = p.Kcrt > 0 ? std::min(p.Kcrt, p.K) : p.K;  // read by the CRT kernels only
    d.Lf = p.f.L;
    d.Lg = p.g.L;
    d.fstride = p.f.stride;
    d.gstride = p.g.stride;
    d.fnc = p.f.nc;
    d.gnc = p.g.nc;
    d.Lout = p.Lout;
    d.mxf = p.f.mx;
    d.mxg = p.g.mx;
    d.f_off = b->in_f[i];
    d.g_off = b->in_g[i];
    d.meta_off = (int64_t)meta.size();
    int start = 0;
    for (int j = 0; j <= p.f.my; ++j) {
      meta.push_back(make_int2(start, p.f.dx[j]));
      start += p.f.dx[j] + 1;
    }
    for (int j = 0; j <= p.g.my; ++j) {
      meta.push_back(make_int2(start, p.g.dx[j]));
      start += p.g.dx[j] + 1;
    }
    d.img_off = b->img_words;
    b->img_words += (int64_t)p.K * d.NI;
    d.out_off = b->out_words;
    b->out_words += (int64_t)p.N * p.Lout;
    const int64_t chunks = (p.Lout + 15) / 16;
    d.xl_off = b->xl_words;
    b->xl_words += (int64_t)p.N * 16 * chunks;
    d.cy_off = b->cy_words;
    b->cy_words += (int64_t)p.N * chunks;
    b->dev_index[i] = (int)b->descs.size();
    b->descs.push_back(d);
    order.push_back(i);
    maxM = std::max(maxM, d.NI / 2);
    maxK = std::max(maxK, p.K);
    maxDx = std::max(maxDx, std::max(p.f.mx, p.g.mx));
    b->info.images += (int64_t)p.K * d.NI;
    b->info.primes_total += p.K;
    b->info.coeffs_total += p.N;
    const double imgs = (double)p.K * d.NI;
    // per image: half of the evaluation (the two images of a point pair share
    // the even and odd parts) plus one product per coefficient to combine them
    if (ctx->cfg.univariate == 1) {  // Schur variant: Horner per coefficient, 4 r (r + 1) products
      const double r = (double)p.f.my + p.g.my;
      b->info.modmul_eval += imgs * ((double)(p.f.my + 1) * (p.f.mx + 1) + (double)(p.g.my + 1) * (p.g.mx + 1));
      b->info.modmul_prs += imgs * 4.0 * r * (r + 1.0);
    } else {
      b->info.modmul_eval += imgs * (0.5 * (p.f.nc + p.g.nc) + (p.f.my + 1) + (p.g.my + 1));
      b->info.modmul_prs += imgs * prs_products(p.f.my, p.g.my);
    }
    b->info.modmul_interp += (double)p.K * ((double)d.NI * d.NI / 2 + 8.0 * d.NI);  // two interpolations of NI / 2
    b->info.modmul_crt += (double)p.N * ((double)d.K * (d.K - 1) + d.K);
  }
  b->shape_off = b->out_words;  // per pair (1 + degree, limbs), written by the last CRT kernel
  b->status_off = b->shape_off + 2 * (int64_t)b->descs.size();
  if (!images_only) b->out_words += 2 * (int64_t)b->descs.size() + 1;  // + the device status word
  if (images_only) b->out_words = std::max(b->out_words, b->img_words);

  // G1 tiles grouped by register-capacity class; costliest pairs first.
  std::sort(order.begin(), order.end(), [&](int x, int y) {
    const PairPlan &a = b->plans[x], &c = b->plans[y];
    double ca = (double)a.K * a.N * (a.f.nc + a.g.nc + 2.0 * a.f.my * a.g.my);
    double cc = (double)c.K * c.N * (c.f.nc + c.g.nc + 2.0 * c.f.my * c.g.my);
    return ca > cc;
  });
  // Tile width and schedule per class: forced by the options or the context,
  // else the tuner's cached choice (timed now when missing and allowed), else
  // 128 points on a persistent grid.
  std::vector<Tile> tiles;
  for (int v = 0; v < 18; ++v) {  // capacities 8 .. 72, with the column and without
    const int cap = 8 * (v / 2 + 1);
    const bool col = v % 2 == 0;
    std::vector<int> members;
    int cmaxN = 0;
    int64_t cimages = 0;
    for (int i : order)
      if (g1_supported_cap(b->plans[i].cap) == cap && rs_g1_column(b->plans[i], cap) == col) {
        members.push_back(i);
        cmaxN = std::max(cmaxN, b->plans[i].N);
        cimages += (int64_t)b->plans[i].K * b->plans[i].N;
      }
    if (members.empty()) continue;
    RsG1Choice ch;
    if (opt.g1_threads > 0) {
      ch.threads = opt.g1_threads;
    } else if (ctx->cfg.tile_points > 0) {
      ch.threads = ctx->cfg.tile_points;
    } else {
      const int64_t key = rs_tune_key(ctx->sms, cap, cmaxN, cimages);
      if (!rs_tune_find(key, &ch) && opt.tune && ctx->cfg.autotune && ctx->cfg.univariate == 0) {
        const int rc = rs_tune_g1(ctx, f, g, b->plans, members, key, &ch);
        if (rc != RS_OK) {
          rs_free_batch(b);
          return rc;
        }
      }
    }
    ch.persistent = (ch.persistent && opt.persistent) ? 1 : 0;
    if (opt.g1_threads > 0 || ctx->cfg.tile_points > 0) ch.persistent = opt.persistent ? 1 : 0;
    const int T = ch.threads;
    RsClassLaunch cl;
    cl.cap = cap;
    cl.col = col;
    cl.threads = T;
    cl.persistent = ch.persistent;
    cl.tile_off = (int64_t)tiles.size();
    // Work items of `run` consecutive chunks of T / 2 point pairs: the block
    // stages a (pair, prime)'s coefficients once per item and walks its
    // chunks.  Runs are as long as the class allows while it keeps at least
    // 16 items per SM for the scheduler to balance.
    int64_t chunks = 0;
    for (int i : members) chunks += (int64_t)b->plans[i].K * (((b->plans[i].N + 1) / 2 + T / 2 - 1) / (T / 2));
    const int run = (int)std::max<int64_t>(1, chunks / (16 * (int64_t)ctx->sms));
    for (int i : members) {
      const PairPlan &p = b->plans[i];
      cl.cost += (double)p.K * p.N * (p.f.nc + p.g.nc + 2.0 * p.f.my * p.g.my);
      cl.smem = std::max(cl.smem, (size_t)rs_g1_smem_words(p, cap, T, col) * 4);
      const int M = (p.N + 1) / 2;  // point pairs: two threads each
      for (int k = 0; k < p.K; ++k) {
        if (ctx->cfg.univariate == 0) {
          for (int x0 = 0; x0 < M; x0 += run * (T / 2))
            tiles.push_back(Tile{b->dev_index[i], k, x0, std::min(run * (T / 2), M - x0)});
        } else {
          for (int x0 = 0; x0 < M; x0 += T / 2) tiles.push_back(Tile{b->dev_index[i], k, x0, std::min(T / 2, M - x0)});
        }
      }
    }
    cl.ntiles = (int)((int64_t)tiles.size() - cl.tile_off);
    if (cl.ntiles > 0) b->classes.push_back(cl);
  }
  std::stable_sort(b->classes.begin(), b->classes.end(),
                   [](const RsClassLaunch &x, const RsClassLaunch &y) { return x.cost > y.cost; });
  if (ctx->cfg.univariate == 1 && !tiles.empty()) {
    b->schur = true;
    b->ntiles_all = (int)tiles.size();
    int rmax = 0;
    size_t staged = 0, fb = 0;
    for (int i : order) {
      const PairPlan &p = b->plans[i];
      const int r = p.f.my + p.g.my;
      rmax = std::max(rmax, r);
      staged = std::max(staged, (size_t)((p.f.my + 1) * (p.f.mx + 1) + (p.g.my + 1) * (p.g.mx + 1)) * 4);
      fb = std::max(fb, (size_t)((size_t)r * r + r + r + 2) * 4);
    }
    b->schur_slots = std::max(1, (rmax + 31) / 32);
    b->schur_smem = staged;
    b->schur_fb_smem = fb;
    if (b->schur_slots > RS_G1S_MAX_SLOTS || staged > 227 * 1024 || fb > 227 * 1024) {
      rs_free_batch(b);
      return rs_fail(ctx, RS_ERR_LIMIT, "Schur variant: m_y + n_y or the staged coefficients exceed its limits");
    }
  }
  std::vector<int2> g2, g3;
  std::vector<int> byN(order);
  std::sort(byN.begin(), byN.end(), [&](int x, int y) { return b->plans[x].N > b->plans[y].N; });
  // G2 launches: the direct form by octaves of point counts, shaped by
  // rs_g2_shape.  Pairs whose transform-based G2 is cheaper go to one launch per transform
  // length instead (256 threads, shared memory 3 N + 2^lg words).
  // The form is chosen per transform-length group: forced by the context or
  // the options, else the tuner's cached choice (timed now when missing and
  // allowed; groups with lg < 7, under 64 point pairs, keep the model's
  // choice), else the model.
  std::vector<int> g2lg(n, 0), g2t_lg(n, 0);  // transform / tensor-core length group per pair
  int bhatK[RS_NTT_LGMAX + 1] = {};
  const bool g2tri = ctx->cfg.g2_form == 3;  // triangular factorisation of the Vandermonde system
  if (g2tri && !images_only && !order.empty()) {
    RsG2Class gc;
    gc.lg = -1;
    gc.off = (int64_t)g2.size();
    int cmaxN = 0;
    for (int i : byN) {
      cmaxN = std::max(cmaxN, b->plans[i].N);
      for (int k = 0; k < b->plans[i].K; ++k) g2.push_back(make_int2(b->dev_index[i], k));
    }
    gc.count = (int)((int64_t)g2.size() - gc.off);
    gc.smem = (size_t)(4 * cmaxN + 97) * 4;
    if (gc.smem > 227 * 1024) {
      rs_free_batch(b);
      return rs_fail(ctx, RS_ERR_LIMIT, "g2_form 3: D + 1 above the shared-memory limit of the form (14,000)");
    }
    b->g2cls.push_back(gc);
  }
  if (!images_only && !g2tri) {
    std::vector<std::vector<int>> bylg(RS_NTT_LGMAX + 1);
    for (int i : byN) {
      const int lg = rs_g2_len((b->plans[i].N + 1) / 2);
      if (lg) bylg[lg].push_back(i);
    }
    for (int lg = 1; lg <= RS_NTT_LGMAX; ++lg) {
      if (bylg[lg].empty()) continue;
      double cd = 0.0, cn = 0.0;
      int64_t images = 0;
      for (int i : bylg[lg]) {
        const PairPlan &p = b->plans[i];
        cd += p.K * rs_g2_cost((p.N + 1) / 2, 0);
        cn += p.K * rs_g2_cost((p.N + 1) / 2, 1);
        images += (int64_t)p.K * p.N;
      }
      const int model = cn < cd ? 1 : 0;
      int form = model;
      if (ctx->cfg.g2_form == 1 || ctx->cfg.g2_form == 2 || ctx->cfg.g2_form == 4) {
        form = ctx->cfg.g2_form == 2 ? 1 : ctx->cfg.g2_form == 4 ? 2 : 0;
      } else if (opt.g2_force >= 0) {
        form = opt.g2_force;
      } else if (lg >= 7) {
        const int64_t key = rs_tune_key_g2(ctx->sms, lg, images);
        RsG1Choice c;
        if (rs_tune_find(key, &c)) {
          form = c.threads;
        } else if (opt.tune && ctx->cfg.autotune) {
          const int rc = rs_tune_g2(ctx, f, g, b->plans, bylg[lg], key, model, &form);
          if (rc != RS_OK) {
            rs_free_batch(b);
            return rc;
          }
        }
      }
      if (!form) continue;
      if (form == 2) {
        for (int i : bylg[lg]) g2t_lg[i] = lg;
        continue;
      }
      for (int i : bylg[lg]) {
        g2lg[i] = lg;
        bhatK[lg] = std::max(bhatK[lg], b->plans[i].K);
      }
    }
  }
  // One tensor-core class over every pair whose length group chose that
  // form: for every prime k, the pairs with K > k in decreasing point count
  // (so a tile's rows have similar lengths), 64 to a row tile
  // (rows 2 slot, 2 slot + 1: even and odd part); a tile's length is its
  // first pair's point-pair count rounded up to 64.  Work items: every 64
  // outputs of every tile, tiles by decreasing length, outputs from the top
  // (the longest items first; a tile's items run close together in time,
  // so its operand digits are read from L2).
  std::vector<G2tTask> g2t_tasks;
  std::vector<G2tRowTile> g2t_rts;
  std::vector<G2tItem> g2t_items;
  int64_t g2t_y_words = 0;
  int g2t_kmax = 0, g2t_tiles = 0;
  b->g2t_x_elems = 0;
  std::vector<int> g2t_mem;
  for (int i : byN)
    if (g2t_lg[i] > 0) g2t_mem.push_back(i);
  if (!images_only && !g2tri && !g2t_mem.empty()) {
    const std::vector<int> &mem = g2t_mem;
    RsG2Class gc;
    gc.lg = g2t_lg[mem[0]];
    gc.tensor = true;
    gc.t_task_off = (int64_t)g2t_tasks.size();
    gc.t_item_off = (int64_t)g2t_items.size();
    const int rt0 = (int)g2t_rts.size();
    int kmax = 0;
    for (int i : mem) kmax = std::max(kmax, b->plans[i].K);
    for (int k = 0; k < kmax; ++k) {
      std::vector<int> rows;
      for (int i : mem)
        if (b->plans[i].K > k) rows.push_back(i);
      for (size_t c0 = 0; c0 < rows.size(); c0 += 64) {
        const int cnt = (int)std::min<size_t>(64, rows.size() - c0);
        G2tRowTile rt;
        memset(&rt, 0, sizeof(rt));
        rt.prime = k;
        rt.mt = (((b->plans[rows[c0]].N + 1) / 2 + 63) / 64) * 64;
        rt.rows = 2 * cnt;
        rt.x_off = b->g2t_x_elems;
        rt.y_off = g2t_y_words;
        b->g2t_x_elems += (int64_t)(rt.mt / 64) * 32768;
        g2t_y_words += (int64_t)128 * rt.mt;
        const int rti = (int)g2t_rts.size();
        g2t_rts.push_back(rt);
        for (int sl = 0; sl < cnt; ++sl) {
          G2tTask t;
          t.pair = b->dev_index[rows[c0 + sl]];
          t.prime = k;
          t.rt = rti;
          t.slot = sl;
          g2t_tasks.push_back(t);
          gc.t_maxM = std::max(gc.t_maxM, (b->plans[rows[c0 + sl]].N + 1) / 2);
        }
        g2t_tiles = std::max(g2t_tiles, rt.mt / 32);
      }
    }
    g2t_kmax = std::max(g2t_kmax, kmax);
    std::vector<int> ord;
    for (int r = rt0; r < (int)g2t_rts.size(); ++r) ord.push_back(r);
    std::stable_sort(ord.begin(), ord.end(), [&](int x, int y) { return g2t_rts[x].mt > g2t_rts[y].mt; });
    for (int r : ord)
      for (int t0 = g2t_rts[r].mt - 64; t0 >= 0; t0 -= 64) g2t_items.push_back(G2tItem{r, t0});
    gc.t_ntask = (int)((int64_t)g2t_tasks.size() - gc.t_task_off);
    gc.t_nitem = (int)((int64_t)g2t_items.size() - gc.t_item_off);
    gc.count = gc.t_ntask;
    b->g2cls.push_back(gc);
  }
  for (int lg = RS_NTT_LGMAX; lg > 0; --lg) {
    if (!bhatK[lg]) continue;
    RsG2Class gc;
    gc.lg = lg;
    gc.off = (int64_t)g2.size();
    int cmaxN = 0;
    for (int i : byN) {
      if (g2lg[i] != lg) continue;
      cmaxN = std::max(cmaxN, (b->plans[i].N + 1) / 2);  // point pairs
      for (int k = 0; k < b->plans[i].K; ++k) g2.push_back(make_int2(b->dev_index[i], k));
    }
    gc.count = (int)((int64_t)g2.size() - gc.off);
    gc.smem = (size_t)(4 * ((cmaxN + 3) & ~3) + 2 * (1 << lg)) * 4;
    b->g2cls.push_back(gc);
  }
  const int nlg = (int)b->g2cls.size();
  if (!g2tri && !images_only) {
    double direct = 0.0;  // the direct form's whole work: a shape is chosen as for that work in tasks of its size
    for (int i : byN)
      if (!g2lg[i] && !g2t_lg[i]) direct += b->plans[i].K * rs_g2_cost((b->plans[i].N + 1) / 2, 0);
    for (size_t u = 0; u < byN.size();) {
      // One launch per octave of point-pair counts, shaped for its largest;
      // octaves of one shape together.  (A shape for every count of an uneven
      // batch of 17 pairs gave 16 launches and 0.36 ms; by octaves 0.27.)
      if (g2lg[byN[u]] || g2t_lg[byN[u]]) {
        ++u;
        continue;
      }
      const int top = (b->plans[byN[u]].N + 1) / 2;
      const RsG2Shape sh = rs_g2_shape(top, (int64_t)(direct / rs_g2_cost(top, 0) + 0.5), ctx->sms, nullptr);
      const RsG2Class *last = (int)b->g2cls.size() > nlg ? &b->g2cls.back() : nullptr;
      if (!last || last->threads != sh.threads || last->halves != sh.halves || last->split != sh.split) {
        RsG2Class nc;
        nc.off = (int64_t)g2.size();
        nc.threads = sh.threads;
        nc.halves = sh.halves;
        nc.split = sh.split;
        b->g2cls.push_back(nc);
      }
      RsG2Class &gc = b->g2cls.back();
      RsG2Shape cur = sh;
      int curM = top;
      for (; u < byN.size(); ++u) {
        const PairPlan &p = b->plans[byN[u]];
        if (g2lg[byN[u]] || g2t_lg[byN[u]]) continue;
        const int M = (p.N + 1) / 2;
        if (2 * M <= top) break;
        if (M != curM) cur = rs_g2_shape(M, (int64_t)(direct / rs_g2_cost(M, 0) + 0.5), ctx->sms, &sh);
        if (cur.halves != sh.halves) break;
        curM = M;
        gc.smem = std::max(gc.smem, cur.smem);
        b->descs[b->dev_index[byN[u]]].g2_seg = cur.seg;
        for (int k = 0; k < p.K; ++k) g2.push_back(make_int2(b->dev_index[byN[u]], k));
      }
      gc.count = (int)((int64_t)g2.size() - gc.off);
    }
  }
  // CRT digits in tiles of 32 coefficients; limbs in blocks of 128
  // coefficients by chunks of 16 output limbs.
  // Digit tiles hold 32 coefficients, or 16 when 32-wide tiles would be
  // fewer than two per SM (few coefficients with many primes each).
  std::vector<int2> g3d;
  std::vector<int4> g3b;  // CRT limb chunks: 128 coefficients x one chunk per block
  // Everything in one kernel (g3f_kernel), one thread per coefficient, for at
  // most 16 primes, and to 80 from 128 coefficients per SM; us before and so:
  // 37 coefficients of 5 primes 13.6 and 9.9, 1,082 of 8 18.1 and 14.1, 129 of 18
  // 20.1 and 20.0, 3,090 of 23 24.9 and 27.2, 10,178 of 42 36 and 48; 51,094 of 9
  // 34.8 and 22.2, 24,994 of 32 52.9 and 36.8, 61,762 of 50 109 and 74, 245,084 of
  // 72 541 and 516.
  // Otherwise, digits: one thread per coefficient when there are enough of them for one
  // each to fill the GPU, the fewer the primes (a thread walks its K^2 / 2
  // products alone): from 96 per SM, 8 K per SM, 1024 per SM for any K.
  // Otherwise tiles of 32 or 16 coefficients on the CUDA cores, the tensor
  // cores in tiles of 128, or, above 256 primes, two levels: tiles for 256
  // digits at a time and their products with the later residues on the tensor
  // cores of all SMs; whichever these times (ms, fitted to the measurements
  // below; 608 schedulers' products against one tile's chain of digit blocks
  // per wave, and for two levels both a group's chain and its waves of far
  // products) say, each with its limbs' time.  Limbs: on the CUDA cores after
  // one thread per coefficient; on the tensor cores after digits there; after
  // tiles on the CUDA cores too, unless a pair has 24 primes and these times
  // say otherwise: a thread's chain over the longest pair's primes or the
  // products of all, against 8 us a block (128 coefficients of a pair and 64
  // limbs, mostly the read-out, however few the coefficients) and 1 us a
  // 64-prime chunk, one block per SM.  With tensor-core limbs from 24 primes on,
  // one long pair took thousands of short ones there.  CRT stage, us, CUDA-core
  // and tensor-core limbs: 4,183 pairs of 97 coefficients and 6 primes with 4 of
  // 1,117 and 116 264 and 467; 1,216 of 55 and 6 with one of 949 and 69 84 and 175;
  // 4,305 of 13 and 52 with 8 of 13 and 790 807 and 891; 359 of 13 and 6 with one
  // of 9 and 63 44 and 51; 288 of 9 and 16 with one of 33 and 219 100 and 59; 822
  // of 9 and 7 with 2 of 9 and 735 675 and 539 (in 70 mixed batches the estimates'
  // choice was at most 6% slower than the other).
  // CRT stage, us: CUDA-core tiles with CUDA-core limbs, with tensor-core
  // limbs, tensor-core digits and limbs, one thread per coefficient (with the
  // digits' earlier kernel, which took one warp through each digit block's 64
  // steps, the first column was 79, 727, 694, 1,650 and 5,910 us in rows 3, 6,
  // 8, 10 and 11):
  //   coefficients  primes (avg)  tiles  + limbs  tensor  per thread
  //     1,160         27             24      22      43      41
  //     3,178          8             24      24      43      30
  //       901         69             46      32      81
  //    18,553         66            132     100     153     360
  //     9,220        310            296     194     247
  //     4,520        514            429     253     383
  //     3,362        436            274     173     297
  //     4,097        546            396     252     403
  //    13,448        436            690     434     368
  //     1,640      1,199            972     542     931
  //     4,520      2,000          4,274   2,223   2,124
  //    16,388        547          1,236     783     500
  //    63,008        526          4,029   2,430   1,784
  //    18,254          7             28      36              22
  //    51,094          9             51      96     239      34
  //    50,782         22             59      76              47
  //    24,994         32             49      53              55
  //   116,878         32            134     170              92
  // Two levels, against the fastest of the others with the carry kernel of
  // kernels_g3.cu: 4,097 of 546 229 -> 184, 4,520 of 514 232 -> 190, 1,640 of
  // 1,199 504 -> 307, 4,520 of 2,000 2,028 -> 1,003, 63,008 of 526 1,792 -> 1,772.
  {
    int64_t nt32 = 0, nt128 = 0, ncoef = 0;
    int kc = 0;  // largest prime count of the Chinese remaindering
    double nk2 = 0.0, limb_work = 0.0, limb_tc = 0.0;  // limbs: products on the CUDA cores; us of blocks on the tensor cores
    for (int i : order) {
      const int K = b->descs[b->dev_index[i]].K, L = b->plans[i].Lout, kb = (K + 63) / 64, units = (L + 63) / 64;
      limb_work += 0.25 * ((b->plans[i].N + 31) / 32) * ((L + 15) / 16) * K;
      // unit u takes about kb - u of the pair's kb chunks: 64 primes are 62 limbs
      limb_tc += (double)((b->plans[i].N + 127) / 128) * (8.0 * units + 0.5 * std::min(kb, units) * (2 * kb + 1 - std::min(kb, units)));
      nt32 += (b->plans[i].N + 31) / 32;
      nt128 += (b->plans[i].N + 127) / 128;
      ncoef += b->plans[i].N;
      kc = std::max(kc, K);
      nk2 += (double)b->plans[i].N * K * K;
    }
    b->g3_kc = kc;
    const int64_t sms = ctx->sms;
    b->g3_jt = nt32 < 2 * sms ? 16 : 32;
    b->g3_perthread = ncoef >= sms * std::min<int64_t>(RS_G3P_MIN_COEF_PER_SM, std::max(96, 8 * kc));
    const double ms_tiles = std::max(1.1e-10 * nk2 * 152 / sms + 0.6e-4 * kc, 2.7e-7 * kc * kc);
    const double ms_tensor = (double)((nt128 + sms - 1) / sms) * kc * 0.55e-3 * (1.0 + kc / 2500.0);
    double ms_two = (kc / 256.0) * std::max(0.037, 0.008 + 0.022 / 16.0 * ncoef / sms);
    for (int c = 4; 64 * c < kc; c += 4) {
      int64_t items = 0;
      for (int i : order) {
        const int kb = (b->descs[b->dev_index[i]].K + 63) / 64;
        if (kb > c) items += (int64_t)((b->plans[i].N + 127) / 128) * (kb - c);
      }
      ms_two += 0.004 + 0.009 * ((items + sms - 1) / sms);
      ++b->g3_nfar;
    }
    b->g3_fused = !images_only && ctx->cfg.crt_form == 0 && kc > 0 &&
                  (kc <= 16 || (kc <= RS_G3F_MAX_K && ncoef >= 128 * sms));
    const bool tc = !b->g3_fused && !b->g3_perthread && !images_only && ctx->cfg.crt_form != 1;
    const double ms_climbs = std::max(2.1e-4 * kc, 2.3e-7 * limb_work * 152 / sms), ms_tlimbs = 1e-3 * limb_tc / sms;
    const bool tlimbs = kc >= RS_G3L_MIN_K && ms_tlimbs < ms_climbs;  // after tiles
    const double ms_cuda = ms_tiles + (tlimbs ? ms_tlimbs : ms_climbs);
    b->g3_two = tc && ctx->cfg.crt_form != 2 && b->g3_nfar > 0 && ms_two + ms_tlimbs < ms_cuda &&
                (kc < RS_G3M_MIN_K || ms_two < ms_tensor);
    if (!b->g3_two) b->g3_nfar = 0;
    b->g3_tensor = tc && !b->g3_two &&
                   (ctx->cfg.crt_form == 2 || (kc >= RS_G3M_MIN_K && ms_tensor + ms_tlimbs < ms_cuda));
    b->g3_tlimbs = tc && (b->g3_tensor || b->g3_two || tlimbs);
  }
  for (int i : order) {
    const PairPlan &p = b->plans[i];
    const int di = b->dev_index[i], chunks = (p.Lout + 15) / 16;
    b->g3_maxL = std::max(b->g3_maxL, p.Lout);
    for (int j = 0; j < p.N; j += 128) g3.push_back(make_int2(di, j));
    for (int j = 0; j < p.N; j += b->g3_jt) g3d.push_back(make_int2(di, j));  // digit tiles
    for (int c = 0; c < chunks; ++c)
      for (int j = 0; j < p.N; j += 128) g3b.push_back(make_int4(di, j, c, 0));
  }
  std::vector<int2> yun;  // square-free factorisation tasks: every (pair, prime), pairs in order
  if (opt.yun_maxm > 0 && !images_only) {
    int maxNp = 1;
    for (int i = 0; i < n; ++i) {
      if (b->dev_index[i] < 0) continue;
      maxNp = std::max(maxNp, b->plans[i].N);
      for (int k = 0; k < b->plans[i].K; ++k) yun.push_back(make_int2(b->dev_index[i], k));
    }
    b->yun_wstride = ((int64_t)maxNp + 3) & ~(int64_t)3;
    b->yun_ostride = ((int64_t)maxNp + 2 * opt.yun_maxm + 2 + 3) & ~(int64_t)3;
  }
  // Tensor-core CRT digits: each task (128 coefficients of a pair) owns its
  // operand digit rows, one 64 KB chunk per 64 of the pair's primes.
  std::vector<int64_t> g3m_xoff;
  b->g3m_x_elems = 0;
  if (b->g3_tlimbs) {
    for (const int2 &t : g3) {
      if (t.y == 0) b->descs[t.x].xd_off = b->g3m_x_elems;
      g3m_xoff.push_back(b->g3m_x_elems);
      b->g3m_x_elems += g3m_tile_elems(b->descs[t.x].K);
    }
  }
  b->nyun = (int)yun.size();
  b->ng2 = images_only ? 0 : (int)g2.size();
  b->ng3 = images_only ? 0 : (int)g3.size();
  b->ng3d = images_only ? 0 : (int)g3d.size();
  b->ng3b = images_only ? 0 : (int)g3b.size();
  b->kmax = maxK;
  b->info.input_bytes = b->in_words * 4;
  b->info.output_bytes = b->out_words * 4;
  b->info.kernel_launches = (b->schur ? 2 : (int64_t)b->classes.size()) + (int64_t)b->g2cls.size() + (b->ng3d > 0) +
                            (b->nyun > 0) +
                            (b->ng3b > 0) +
                            (b->ng3 > 0);
  if (b->g3_fused) b->info.kernel_launches -= (b->ng3d > 0) + (b->ng3b > 0);
  b->info.kernel_launches += b->g3_two ? b->g3_nfar + (b->g3_kc + 255) / 256 - 1 : 0;
  for (const auto &gc : b->g2cls)
    if (gc.tensor) b->info.kernel_launches += 4;  // five launches per tensor-core class

  int rc = RS_OK;
  if (!order.empty()) rc = rs_ensure_tables(ctx, maxK, maxM, maxDx);
  for (int lg = 1; lg <= RS_NTT_LGMAX && rc == RS_OK; ++lg)
    if (bhatK[lg]) rc = rs_ensure_bhat(ctx, lg, bhatK[lg]);
  if (rc == RS_OK && g2t_kmax > 0) rc = rs_ensure_g2t_btile(ctx, g2t_kmax, g2t_tiles);
  if (rc == RS_OK && (b->g3_tensor || b->g3_two)) rc = rs_ensure_g3m_wtiles(ctx, (maxK + 63) / 64);
  if (rc == RS_OK && b->g3_tlimbs) rc = rs_ensure_g3l_tiles(ctx, (maxK + 63) / 64);
  if (rc == RS_OK && b->g3_tlimbs) {
    // The limbs then come from the tensor cores too: one task per (digit
    // task, unit of 64 limbs) instead of the limb chunks, with the chunks
    // from the first whose prefix products reach the unit; the longest first.
    std::vector<int32_t> cb;
    {
      std::lock_guard<std::mutex> lock(ctx->tab_mu);
      cb = ctx->h_g3l_cbase;
    }
    const int KBt = (int)cb.size() - 1;
    std::vector<std::pair<int, int4>> lt;
    for (size_t ti = 0; ti < g3.size(); ++ti) {
      const PairDesc &pd = b->descs[g3[ti].x];
      const int KBp = (pd.K + 63) / 64, units = (pd.Lout + 63) / 64;
      int lo = 0;
      for (int u = 0; u < units; ++u) {
        while (lo < KBt && cb[lo + 1] - cb[lo] - 1 < u) ++lo;
        lt.push_back({KBp > lo ? KBp - lo : 0, make_int4((int)ti, u, lo, 0)});
      }
    }
    std::stable_sort(lt.begin(), lt.end(), [](const std::pair<int, int4> &x, const std::pair<int, int4> &y) {
      return x.first > y.first;
    });
    g3b.clear();
    for (const auto &x : lt) g3b.push_back(x.second);
    b->ng3b = (int)g3b.size();
  }
  if (rc != RS_OK) {
    rs_free_batch(b);
    return rc;
  }
  DevGuard dg(ctx->device);
  size_t off = 0;  // one device arena carved into every buffer of the batch
  auto carve = [&](size_t bytes) {
    size_t o = off;
    off += align_up(bytes);
    return o;
  };
  const size_t o_in = carve(b->in_words * 4), o_meta = carve(meta.size() * sizeof(int2)),
               o_pairs = carve(b->descs.size() * sizeof(PairDesc)), o_tiles = carve(tiles.size() * sizeof(Tile)),
               o_num = carve(b->img_words * 4), o_den = carve(b->img_words * 4),
               o_xl = carve(std::max(b->xl_words, b->out_words) * 4), o_out = carve(b->out_words * 4),
               // after the results' shapes and status word: all that a pass zeroes, in one piece
               o_cnt = carve(RS_G1_COUNTERS * sizeof(int32_t)), o_st = carve(ST_COUNT * sizeof(unsigned long long)),
               o_g2 = carve(g2.size() * sizeof(int2)), o_g3 = carve(g3.size() * sizeof(int2)),
               o_cy = carve(b->cy_words * 8),
               o_g3d = carve(g3d.size() * sizeof(int2)), o_yt = carve(yun.size() * sizeof(int2)),
               o_yo = carve((size_t)b->nyun * b->yun_ostride * 4), o_yw = carve((size_t)b->nyun * 8 * b->yun_wstride * 4),
               o_g3b = carve(g3b.size() * sizeof(int4)), o_fail = carve(b->schur ? b->img_words * sizeof(int2) : 0),
               o_tt = carve(g2t_tasks.size() * sizeof(G2tTask)), o_trt = carve(g2t_rts.size() * sizeof(G2tRowTile)),
               o_tit = carve(g2t_items.size() * sizeof(G2tItem)), o_tx = carve(b->g2t_x_elems * sizeof(uint16_t)),
               o_ty = carve(g2t_y_words * 4), o_g3mx = carve(b->g3m_x_elems * sizeof(uint16_t)),
               o_g3mo = carve(g3m_xoff.size() * sizeof(int64_t));
  cudaError_t e = opt.stream_ordered ? cudaMallocAsync(&b->arena, off, b->stream) : cudaMalloc(&b->arena, off);
  if (e != cudaSuccess) {
    b->arena = nullptr;
    rs_free_batch(b);
    return rs_fail(ctx, rs_cuda_code(e), std::string("device arena: ") + cudaGetErrorString(e));
  }
  char *base = static_cast<char *>(b->arena);
  b->d_in = (uint32_t *)(base + o_in);
  b->d_meta = (int2 *)(base + o_meta);
  b->d_pairs = (PairDesc *)(base + o_pairs);
  b->d_tiles = (Tile *)(base + o_tiles);
  b->d_counters = (int32_t *)(base + o_cnt);
  b->d_num = (uint32_t *)(base + o_num);
  b->d_den = (uint32_t *)(base + o_den);
  b->d_xl = (uint32_t *)(base + o_xl);
  b->d_out = (uint32_t *)(base + o_out);
  b->d_g2 = (int2 *)(base + o_g2);
  b->d_g3 = (int2 *)(base + o_g3);
  b->d_stats = (unsigned long long *)(base + o_st);
  b->d_cy = (int64_t *)(base + o_cy);
  b->d_g3d = (int2 *)(base + o_g3d);
  b->d_yun_tasks = (int2 *)(base + o_yt);
  b->d_yun_out = (uint32_t *)(base + o_yo);
  b->d_yun_work = (uint32_t *)(base + o_yw);
  b->d_g3b = (int4 *)(base + o_g3b);
  b->d_fail = b->schur ? (int2 *)(base + o_fail) : nullptr;
  b->d_g2t_tasks = (G2tTask *)(base + o_tt);
  b->d_g2t_rts = (G2tRowTile *)(base + o_trt);
  b->d_g2t_items = (G2tItem *)(base + o_tit);
  b->d_g2t_x = (uint16_t *)(base + o_tx);
  b->d_g2t_y = (uint32_t *)(base + o_ty);
  b->d_g3m_x = (uint16_t *)(base + o_g3mx);
  b->d_g3m_xoff = (int64_t *)(base + o_g3mo);
  // Tensor-core operand digits: rows and inputs beyond each pair's points
  // stay zero for the batch's life (the kernels write only inputs < M).
  if (b->g3m_x_elems) e = cudaMemsetAsync(b->d_g3m_x, 0, b->g3m_x_elems * sizeof(uint16_t), b->stream);
  if (e == cudaSuccess && b->g2t_x_elems)
    e = cudaMemsetAsync(b->d_g2t_x, 0, b->g2t_x_elems * sizeof(uint16_t), b->stream);
  if (e != cudaSuccess) {
    rs_free_batch(b);
    return rs_fail(ctx, rs_cuda_code(e), std::string("tensor-core operands: ") + cudaGetErrorString(e));
  }

  if (opt.h_in && opt.h_in_words >= b->in_words && opt.h_out && opt.h_out_words >= b->out_words) {
    b->h_in = opt.h_in;
    b->h_out = opt.h_out;
  } else {
    b->own_host = true;
    if (b->in_words && cudaMallocHost((void **)&b->h_in, b->in_words * 4) != cudaSuccess) rc = RS_ERR_NOMEM;
    if (rc == RS_OK && b->out_words && cudaMallocHost((void **)&b->h_out, b->out_words * 4) != cudaSuccess)
      rc = RS_ERR_NOMEM;
    if (rc != RS_OK) {
      rs_free_batch(b);
      return rs_fail(ctx, rc, "cudaMallocHost (staging)");
    }
  }
  // Static per-batch tables, ordered on the batch stream.  With borrowed
  // pinned staging large enough they are packed behind the inputs and copied
  // without waiting; otherwise they are copied from pageable memory and the
  // stream is synchronised before the host vectors go away.
  struct Piece {
    void *dst;
    const void *src;
    size_t bytes;
  };
  const Piece pieces[] = {{b->d_meta, meta.data(), meta.size() * sizeof(int2)},
                          {b->d_pairs, b->descs.data(), b->descs.size() * sizeof(PairDesc)},
                          {b->d_tiles, tiles.data(), tiles.size() * sizeof(Tile)},
                          {b->d_g2, g2.data(), g2.size() * sizeof(int2)},
                          {b->d_g3, g3.data(), g3.size() * sizeof(int2)},
                          {b->d_g3d, g3d.data(), g3d.size() * sizeof(int2)},
                          {b->d_yun_tasks, yun.data(), yun.size() * sizeof(int2)},
                          {b->d_g3b, g3b.data(), g3b.size() * sizeof(int4)},
                          {b->d_g2t_tasks, g2t_tasks.data(), g2t_tasks.size() * sizeof(G2tTask)},
                          {b->d_g2t_rts, g2t_rts.data(), g2t_rts.size() * sizeof(G2tRowTile)},
                          {b->d_g2t_items, g2t_items.data(), g2t_items.size() * sizeof(G2tItem)},
                          {b->d_g3m_xoff, g3m_xoff.data(), g3m_xoff.size() * sizeof(int64_t)}};
  size_t static_bytes = 0;
  for (const Piece &pc : pieces) static_bytes += (pc.bytes + 15) & ~(size_t)15;
  const bool pinned_static = !b->own_host && (size_t)opt.h_in_words * 4 >= (size_t)b->in_words * 4 + static_bytes;
  char *stage = pinned_static ? reinterpret_cast<char *>(b->h_in + b->in_words) : nullptr;
  for (const Piece &pc : pieces) {
    if (rc != RS_OK || pc.bytes == 0) continue;
    const void *src = pc.src;
    if (stage) {
      memcpy(stage, pc.src, pc.bytes);
      src = stage;
      stage += (pc.bytes + 15) & ~(size_t)15;
    }
    cudaError_t e2 = cudaMemcpyAsync(pc.dst, src, pc.bytes, cudaMemcpyHostToDevice, b->stream);
    if (e2 != cudaSuccess) rc = rs_fail(ctx, RS_ERR_CUDA, std::string("cudaMemcpyAsync: ") + cudaGetErrorString(e2));
  }
  if (rc == RS_OK && !pinned_static) {
    cudaError_t e2 = cudaStreamSynchronize(b->stream);
    if (e2 != cudaSuccess) rc = rs_fail(ctx, RS_ERR_CUDA, std::string("sync: ") + cudaGetErrorString(e2));
  }
  {
    // Kernel attributes and occupancies, once per context.
    std::lock_guard<std::mutex> lock(ctx->prep_mu);
    if (rc == RS_OK && nlg > 0 && !ctx->g2n_ready) {
      cudaError_t e2 = g2n_prepare();
      if (e2 != cudaSuccess) rc = rs_fail(ctx, RS_ERR_CUDA, std::string("G2 set-up: ") + cudaGetErrorString(e2));
      ctx->g2n_ready = e2 == cudaSuccess;
    }
    if (rc == RS_OK && (b->g3_tensor || b->g3_two) && !ctx->g3m_ready) {
      cudaError_t e2 = g3m_prepare();
      if (e2 != cudaSuccess) rc = rs_fail(ctx, RS_ERR_CUDA, std::string("G3 set-up: ") + cudaGetErrorString(e2));
      ctx->g3m_ready = e2 == cudaSuccess;
    }
    if (rc == RS_OK && b->g3_tlimbs && !ctx->g3l_ready) {
      cudaError_t e2 = g3l_prepare();
      if (e2 != cudaSuccess) rc = rs_fail(ctx, RS_ERR_CUDA, std::string("G3 set-up: ") + cudaGetErrorString(e2));
      ctx->g3l_ready = e2 == cudaSuccess;
    }
    if (rc == RS_OK && g2t_kmax > 0 && !ctx->g2t_ready) {
      cudaError_t e2 = g2t_prepare();
      if (e2 != cudaSuccess) rc = rs_fail(ctx, RS_ERR_CUDA, std::string("G2 set-up: ") + cudaGetErrorString(e2));
      ctx->g2t_ready = e2 == cudaSuccess;
    }
    if (rc == RS_OK && !b->g2cls.empty() && !ctx->g2_ready) {
      cudaError_t e2 = g2_prepare();
      if (e2 != cudaSuccess) rc = rs_fail(ctx, RS_ERR_CUDA, std::string("G2 set-up: ") + cudaGetErrorString(e2));
      ctx->g2_ready = e2 == cudaSuccess;
    }
    if (rc == RS_OK && b->g3_fused && !ctx->g3f_ready) {
      cudaError_t e2 = g3f_prepare();
      if (e2 != cudaSuccess) rc = rs_fail(ctx, RS_ERR_CUDA, std::string("CRT set-up: ") + cudaGetErrorString(e2));
      ctx->g3f_ready = e2 == cudaSuccess;
    }
    for (auto &cl : b->classes) {
      if (rc != RS_OK) break;
      const int64_t key = ((int64_t)cl.cap << 40) | ((int64_t)cl.col << 39) | ((int64_t)cl.threads << 24) | (int64_t)((cl.smem + 1023) / 1024);
      auto it = ctx->g1_occupancy.find(key);
      int mb = 0;
      if (it != ctx->g1_occupancy.end()) {
        mb = it->second;
      } else {
        cudaError_t e2 = g1_prepare(cl.cap, cl.col, cl.threads, ((cl.smem + 1023) / 1024) * 1024, &mb);
        if (e2 != cudaSuccess) {
          rc = rs_fail(ctx, RS_ERR_CUDA, std::string("G1 set-up: ") + cudaGetErrorString(e2));
          break;
        }
        ctx->g1_occupancy[key] = mb;
      }
      if (mb < 1) mb = 1;
      cl.blocks = cl.persistent ? std::min(cl.ntiles, mb * ctx->sms) : cl.ntiles;
    }
  }
  if (ctx->cfg.timing || opt.timing)
    for (auto &ev : b->ev)
      if (rc == RS_OK && cudaEventCreate(&ev) != cudaSuccess) rc = rs_fail(ctx, RS_ERR_CUDA, "cudaEventCreate");
  if (opt.fork && (b->classes.size() > 1 || b->g2cls.size() > 1)) {
    b->jev.assign(b->classes.size() + b->g2cls.size(), nullptr);
    for (auto &ev : b->fev)
      if (rc == RS_OK && cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess)
        rc = rs_fail(ctx, RS_ERR_CUDA, "cudaEventCreate");
    for (auto &ev : b->jev)
      if (rc == RS_OK && cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess)
        rc = rs_fail(ctx, RS_ERR_CUDA, "cudaEventCreate");
  }
  if (rc != RS_OK) {
    rs_free_batch(b);
    return rc;
  }
  *out = b;
  return RS_OK;
}

int rs_upload(rs_batch *b, const rs_bipoly *f, const rs_bipoly *g) {
  rs_ctx *ctx = b->ctx;
  // one thread copies about 10 GB/s: shared from 256 KiB on
  const int threads = (int)std::min<int64_t>(16, b->in_words >> 15);
  const int step = std::max(1, b->n / 64);
  ctx->pool.run((b->n + step - 1) / step, threads, [&](int t) {
    for (int i = t * step; i < std::min(b->n, (t + 1) * step); ++i) {
      const PairPlan &p = b->plans[i];
      if (p.status != RS_OK || p.trivial_zero) continue;
      memcpy(b->h_in + b->in_f[i], f[i].coeffs, rs_used_words(p, p.f) * 4);
      memcpy(b->h_in + b->in_g[i], g[i].coeffs, rs_used_words(p, p.g) * 4);
    }
  });
  if (b->in_words)
    RS_CUDA(ctx, cudaMemcpyAsync(b->d_in, b->h_in, b->in_words * 4, cudaMemcpyHostToDevice, b->stream));
  return RS_OK;
}

static cudaError_t record(cudaEvent_t e, cudaStream_t s, bool capturing) {
  return capturing ? cudaEventRecordWithFlags(e, s, cudaEventRecordExternal) : cudaEventRecord(e, s);
}

// The launches of one stage are independent (disjoint tiles or tasks): with
// fork events they run as parallel branches on the context's side streams
// (inside a captured graph: parallel graph nodes), so the tail of one launch
// overlaps the next instead of idling SMs.  Branch i of the stage uses side
// stream i mod 8 and join event j0 + i.
static cudaStream_t branch_begin(rs_batch *b, int stage, int i, cudaStream_t s, cudaError_t *e) {
  if (!b->fev[stage]) return s;
  cudaStream_t si = b->ctx->side[i % 8];
  if (*e == cudaSuccess && i == 0) *e = cudaEventRecord(b->fev[stage], s);
  if (*e == cudaSuccess) *e = cudaStreamWaitEvent(si, b->fev[stage], 0);
  return si;
}

static void branch_end(rs_batch *b, int stage, int j, cudaStream_t si, cudaError_t *e) {
  if (!b->fev[stage]) return;
  if (*e == cudaSuccess) *e = cudaEventRecord(b->jev[j], si);
}

static void join_all(rs_batch *b, int stage, int j0, int n, cudaStream_t s, cudaError_t *e) {
  if (!b->fev[stage]) return;
  for (int j = j0; j < j0 + n && *e == cudaSuccess; ++j) *e = cudaStreamWaitEvent(s, b->jev[j], 0);
}

static int enqueue(rs_batch *b, bool capturing) {
  rs_ctx *ctx = b->ctx;
  cudaStream_t s = b->stream;
  const bool timing = ctx->cfg.timing != 0 || b->opt.timing;
  RsTables tab;
  {
    std::lock_guard<std::mutex> lock(ctx->tab_mu);
    tab = ctx->tab;
  }
  // Counters and statistics, and before them the results' shapes and status
  // word: one launch (four of them were 4 us of a small call's 46).
  char *const z0 = b->opt.images_only ? (char *)b->d_counters : (char *)(b->d_out + b->shape_off);
  RS_CUDA(ctx, cudaMemsetAsync(z0, 0, (size_t)((char *)(b->d_stats + ST_COUNT) - z0), s));
  if (timing) RS_CUDA(ctx, record(b->ev[0], s, capturing));
  if (b->schur) {  // Schur variant of G1 over every tile, then the elimination fallback
    G1sArgs a;
    a.pairs = b->d_pairs;
    a.tiles = b->d_tiles;
    a.limbs = b->d_in;
    a.mods = ctx->d_mods;
    a.vtab = ctx->d_vtab;
    a.qp = tab.qp;
    a.tstride = tab.cstride;
    a.num = b->d_num;
    a.den = b->d_den;
    a.fail = b->d_fail;
    a.fail_count = b->d_counters + RS_G1_COUNTERS - 1;
    a.stats = b->d_stats;
    RS_CUDA(ctx, launch_g1s(b->schur_slots, b->ntiles_all, b->schur_smem, a, s));
    RS_CUDA(ctx, launch_g1s_fallback(2 * ctx->sms, b->schur_fb_smem, a, s));
  }
  int ci = 0;
  for (const auto &cl : b->classes) {
    if (b->schur) break;
    G1Args a;
    a.pairs = b->d_pairs;
    a.tiles = b->d_tiles + cl.tile_off;
    a.ntiles = cl.ntiles;
    a.persistent = cl.persistent;
    a.counter = b->d_counters + (ci++);
    a.limbs = b->d_in;
    a.meta = b->d_meta;
    a.mods = ctx->d_mods;
    a.qc = tab.qc;
    a.qn = tab.qn;
    a.qp = tab.qp;
    a.tstride = tab.cstride;
    a.vtab = ctx->d_vtab;
    a.num = b->d_num;
    a.den = b->d_den;
    a.stats = b->d_stats;
    cudaError_t fe = cudaSuccess;
    cudaStream_t si = branch_begin(b, 0, ci - 1, s, &fe);
    RS_CUDA(ctx, fe);
    RS_CUDA(ctx, launch_g1(cl.cap, cl.col, cl.threads, cl.blocks, cl.smem, a, si));
    branch_end(b, 0, ci - 1, si, &fe);
    RS_CUDA(ctx, fe);
  }
  {
    cudaError_t fe = cudaSuccess;
    if (!b->schur) join_all(b, 0, 0, (int)b->classes.size(), s, &fe);
    RS_CUDA(ctx, fe);
  }
  if (timing) RS_CUDA(ctx, record(b->ev[1], s, capturing));
  uint32_t *bhat[RS_NTT_LGMAX + 1];
  {
    std::lock_guard<std::mutex> lock(ctx->tab_mu);
    for (int l = 0; l <= RS_NTT_LGMAX; ++l) bhat[l] = ctx->bhat[l];
  }
  uint16_t *g2t_bt = nullptr;
  int g2t_tiles = 0;
  {
    std::lock_guard<std::mutex> lock(ctx->tab_mu);
    g2t_bt = ctx->g2t_bt;
    g2t_tiles = ctx->g2t_tiles;
  }
  int gi = 0;
  for (const auto &gc : b->g2cls) {
    if (gc.tensor) {
      G2tArgs at;
      at.pairs = b->d_pairs;
      at.tasks = b->d_g2t_tasks + gc.t_task_off;
      at.rts = b->d_g2t_rts;
      at.items = b->d_g2t_items + gc.t_item_off;
      at.mods = ctx->d_mods;
      at.num = b->d_num;
      at.den = b->d_den;
      at.coef = b->d_num;
      at.finv = tab.finv;
      at.gtab = tab.gtab;
      at.hq = tab.hq;
      at.tab_stride = tab.N;
      at.btile = g2t_bt;
      at.bt_tiles = g2t_tiles;
      at.x = b->d_g2t_x;
      at.y = b->d_g2t_y;
      at.err = reinterpret_cast<int32_t *>(b->d_out + b->status_off);
      at.stall = ctx->d_stall;
      const int j = (int)b->classes.size() + gi;
      cudaError_t fe = cudaSuccess;
      cudaStream_t si = branch_begin(b, 1, gi, s, &fe);
      RS_CUDA(ctx, fe);
      RS_CUDA(ctx, launch_g2t(gc.t_ntask, gc.t_nitem, gc.t_maxM, at, si));
      branch_end(b, 1, j, si, &fe);
      RS_CUDA(ctx, fe);
      ++gi;
      continue;
    }
    if (gc.lg < 0) {
      G2sArgs as;
      as.pairs = b->d_pairs;
      as.tasks = b->d_g2 + gc.off;
      as.mods = ctx->d_mods;
      as.num = b->d_num;
      as.den = b->d_den;
      as.coef = b->d_num;
      as.qp = tab.qp;
      as.tstride = tab.cstride;
      const int j = (int)b->classes.size() + gi;
      cudaError_t fe = cudaSuccess;
      cudaStream_t si = branch_begin(b, 1, gi, s, &fe);
      RS_CUDA(ctx, fe);
      RS_CUDA(ctx, launch_g2s(gc.count, gc.smem, as, si));
      branch_end(b, 1, j, si, &fe);
      RS_CUDA(ctx, fe);
      ++gi;
      continue;
    }
    if (gc.lg > 0) {
      G2nArgs an;
      an.pairs = b->d_pairs;
      an.tasks = b->d_g2 + gc.off;
      an.mods = ctx->d_mods;
      an.num = b->d_num;
      an.den = b->d_den;
      an.coef = b->d_num;
      an.finv = tab.finv;
      an.hq = tab.hq;
      an.gtab = tab.gtab;
      an.tab_stride = tab.N;
      an.tw = ctx->d_ntt_tw;
      an.bhat = bhat[gc.lg];
      an.nc = ctx->nttc;
      an.lg = gc.lg;
      const int j = (int)b->classes.size() + gi;
      cudaError_t fe = cudaSuccess;
      cudaStream_t si = branch_begin(b, 1, gi, s, &fe);
      RS_CUDA(ctx, fe);
      RS_CUDA(ctx, launch_g2n(gc.count, gc.smem, an, si));
      branch_end(b, 1, j, si, &fe);
      RS_CUDA(ctx, fe);
      ++gi;
      continue;
    }
    G2Args a2;
    a2.pairs = b->d_pairs;
    a2.tasks = b->d_g2 + gc.off;
    a2.mods = ctx->d_mods;
    a2.num = b->d_num;
    a2.den = b->d_den;
    a2.coef = b->d_num;
    a2.finv = tab.finv;
    a2.hq = tab.hq;
    a2.gtab = tab.gtab;
    a2.btab = tab.btab;
    a2.tab_stride = tab.N;
    a2.halves = gc.halves;
    a2.split = gc.split;
    const int j = (int)b->classes.size() + gi;
    cudaError_t fe = cudaSuccess;
    cudaStream_t si = branch_begin(b, 1, gi, s, &fe);
    RS_CUDA(ctx, fe);
    RS_CUDA(ctx, launch_g2(gc.threads, gc.count, gc.smem, a2, si));
    branch_end(b, 1, j, si, &fe);
    RS_CUDA(ctx, fe);
    ++gi;
  }
  {
    cudaError_t fe = cudaSuccess;
    join_all(b, 1, (int)b->classes.size(), (int)b->g2cls.size(), s, &fe);
    RS_CUDA(ctx, fe);
  }
  if (b->nyun) {  // square-free factorisation of R mod p, before G3 overwrites the residues
    if (timing) RS_CUDA(ctx, record(b->ev[4], s, capturing));
    YunArgs ya;
    ya.pairs = b->d_pairs;
    ya.tasks = b->d_yun_tasks;
    ya.mods = ctx->d_mods;
    ya.coef = b->d_num;
    ya.out = b->d_yun_out;
    ya.work = b->d_yun_work;
    ya.ostride = b->yun_ostride;
    ya.wstride = b->yun_wstride;
    ya.maxm = b->opt.yun_maxm;
    RS_CUDA(ctx, launch_yun(b->nyun, ya, s));
  }
  if (timing) RS_CUDA(ctx, record(b->ev[2], s, capturing));
  if (b->ng3) {
    G3Args a3;
    a3.pairs = b->d_pairs;
    a3.tasks = b->d_g3;
    a3.ctasks = b->d_g3b;
    a3.mods = ctx->d_mods;
    a3.crt = ctx->d_crt;
    a3.wtab = tab.wtab;
    a3.wtri = tab.wtri;
    a3.p16 = tab.p16;
    a3.poff = tab.poff;
    a3.nh = tab.nh;
    a3.coef = b->d_num;
    a3.xl = b->d_xl;
    a3.carry = b->d_cy;
    a3.out = b->d_out;
    a3.shape = reinterpret_cast<int32_t *>(b->d_out + b->shape_off);
    a3.kmax = b->kmax;
    a3.signed_digits = b->g3_tlimbs ? 1 : 0;
    a3.xdig = b->g3_tlimbs ? b->d_g3m_x : nullptr;
    if (b->g3_fused) {
      RS_CUDA(ctx, launch_g3f(b->ng3, b->g3_kc, a3, b->d_g3, s));
    } else if (b->g3_perthread) {
      RS_CUDA(ctx, launch_g3p(b->ng3, a3, b->d_g3, s));
    } else if (b->g3_tensor) {
      G3mArgs am;
      am.pairs = b->d_pairs;
      am.tasks = b->d_g3;
      am.mods = ctx->d_mods;
      am.crt = ctx->d_crt;
      am.wtab = tab.wtab;
      {
        std::lock_guard<std::mutex> lock(ctx->tab_mu);
        am.wtiles = ctx->g3m_wt;
        am.rtiles = ctx->g3m_rt;
      }
      am.coef = b->d_num;
      am.xdig = b->d_g3m_x;
      am.xoff = b->d_g3m_xoff;
      am.err = reinterpret_cast<int32_t *>(b->d_out + b->status_off);
      am.stall = ctx->d_stall;
      RS_CUDA(ctx, launch_g3m(b->ng3, am, s));
    } else if (b->g3_two) {
      // groups of four digit blocks: their digits, then their products with the rest
      G3uArgs au;
      au.pairs = b->d_pairs;
      au.tasks = b->d_g3;
      au.mods = ctx->d_mods;
      {
        std::lock_guard<std::mutex> lock(ctx->tab_mu);
        au.wtiles = ctx->g3m_wt;
      }
      au.coef = b->d_num;
      au.xdig = b->d_g3m_x;
      au.xoff = b->d_g3m_xoff;
      au.ntasks = b->ng3;
      au.err = reinterpret_cast<int32_t *>(b->d_out + b->status_off);
      au.stall = ctx->d_stall;
      const int KB = (b->g3_kc + 63) / 64;
      for (int c = 0; c < KB; c += 4) {
        a3.kbeg = 64 * c;
        a3.kend = 64 * (c + 4);
        RS_CUDA(ctx, launch_g3t(b->ng3d, a3, b->d_g3d, s, b->g3_jt));
        au.c0 = c;
        au.c1 = c + 4;
        au.nkb = KB - au.c1;
        if (au.nkb > 0) RS_CUDA(ctx, launch_g3u(ctx->sms, au, s));
      }
    } else {
      RS_CUDA(ctx, launch_g3t(b->ng3d, a3, b->d_g3d, s, b->g3_jt));
    }
    if (b->g3_tlimbs) {
      G3lArgs al;
      al.pairs = b->d_pairs;
      al.tasks = b->d_g3;
      al.ltasks = b->d_g3b;
      al.xdig = b->d_g3m_x;
      al.xoff = b->d_g3m_xoff;
      {
        std::lock_guard<std::mutex> lock(ctx->tab_mu);
        al.btiles = ctx->g3l_bt;
        al.cbase = ctx->g3l_cbase;
      }
      al.xl = b->d_xl;
      al.carry = b->d_cy;
      al.err = reinterpret_cast<int32_t *>(b->d_out + b->status_off);
      al.stall = ctx->d_stall;
      RS_CUDA(ctx, launch_g3l(b->ng3b, al, s));
    }
    // the output kernel; the limb chunks unless the tensor cores formed the limbs
    if (!b->g3_fused)
      RS_CUDA(ctx, launch_g3bc(b->g3_tlimbs ? 0 : b->ng3b, b->ng3, b->g3_maxL, ctx->sms, a3, b->d_g3, s));
  }
  if (timing) RS_CUDA(ctx, record(b->ev[3], s, capturing));
  return RS_OK;
}

int rs_run(rs_batch *b) {
  rs_ctx *ctx = b->ctx;
  DevGuard dg(ctx->device);
  if (b->opt.use_graph && !b->opt.images_only) {
    if (!b->gexec) {
      RS_CUDA(ctx, cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal));
      int rc = enqueue(b, true);
      cudaGraph_t graph = nullptr;
      cudaError_t e = cudaStreamEndCapture(b->stream, &graph);
      if (rc != RS_OK) {
        if (graph) cudaGraphDestroy(graph);
        return rc;
      }
      if (e != cudaSuccess) return rs_fail(ctx, RS_ERR_CUDA, std::string("graph capture: ") + cudaGetErrorString(e));
      e = cudaGraphInstantiate(&b->gexec, graph, 0);
      cudaGraphDestroy(graph);
      if (e != cudaSuccess) return rs_fail(ctx, RS_ERR_CUDA, std::string("graph instantiate: ") + cudaGetErrorString(e));
    }
    RS_CUDA(ctx, cudaGraphLaunch(b->gexec, b->stream));
  } else {
    int rc = enqueue(b, false);
    if (rc != RS_OK) return rc;
  }
  b->ran = true;
  return RS_OK;
}

int rs_fetch_async(rs_batch *b) {
  rs_ctx *ctx = b->ctx;
  if (!b->ran) return rs_fail(ctx, RS_ERR_STATE, "batch has not been run");
  if (b->out_words)
    RS_CUDA(ctx, cudaMemcpyAsync(b->h_out, b->d_out, b->out_words * 4, cudaMemcpyDeviceToHost, b->stream));
  return RS_OK;
}

// Degree and limb count of pair i's result (recorded on the device by the
// last CRT kernel and copied back with the limbs), and its limbs in the host
// staging buffer.
static const uint32_t *result_shape(rs_batch *b, int i, int *deg, int *limbs) {
  const PairPlan &p = b->plans[i];
  *deg = -1;
  *limbs = 1;
  if (p.trivial_zero) return nullptr;
  const int d = b->dev_index[i];
  const int32_t *shape = reinterpret_cast<const int32_t *>(b->h_out + b->shape_off) + 2 * (size_t)d;
  *deg = shape[0] - 1;
  *limbs = std::max(1, (int)shape[1]);
  return b->h_out + b->descs[d].out_off;
}

// The device status word copied back with the results: non-zero when a
// bounded wait of the tensor-core interpolation ran out in the last run.
static int device_status(rs_batch *b) {
  if ((b->g2t_x_elems == 0 && !b->g3_tlimbs) || b->out_words <= b->status_off || !b->h_out) return RS_OK;
  return b->h_out[b->status_off] ? RS_ERR_TIMEOUT : RS_OK;
}

int rs_unpack_one(rs_batch *b, int i, std::vector<uint32_t> &words, int *deg, int *limbs) {
  const PairPlan &p = b->plans[i];
  if (p.status != RS_OK) return p.status;
  if (device_status(b) != RS_OK) return RS_ERR_TIMEOUT;
  const uint32_t *w = result_shape(b, i, deg, limbs);
  try {
    words.clear();
    words.reserve((size_t)(*deg + 1) * *limbs);
    for (int j = 0; j <= *deg; ++j) words.insert(words.end(), w + (size_t)j * p.Lout, w + (size_t)j * p.Lout + *limbs);
  } catch (const std::exception &) {
    return RS_ERR_NOMEM;
  }
  return RS_OK;
}

// Shape of pair i's result into o, and whether its limbs can be copied there.
static int shape_pair(rs_batch *b, int i, rs_upoly &o) {
  const PairPlan &p = b->plans[i];
  int rc = p.status;
  if (rc == RS_OK && !o.coeffs && o.capacity_words > 0) rc = RS_ERR_ARG;
  if (rc != RS_OK) return rc;
  int deg, L;
  result_shape(b, i, &deg, &L);
  o.deg = deg;
  o.limbs = L;
  return (int64_t)(deg + 1) * L > o.capacity_words ? RS_ERR_CAPACITY : RS_OK;
}

// Results to the caller's buffers: the shapes (and the status word) are copied
// back first, then the limbs in pieces; while one piece is on its way the host
// threads trim and copy the one before out of the staging buffer.
static int fetch(rs_batch *b, rs_upoly *out, int32_t *status) {
  rs_ctx *ctx = b->ctx;
  DevGuard dg(ctx->device);
  if (!b->ran) return rs_fail(ctx, RS_ERR_STATE, "batch has not been run");
  const int n = b->n;
  const int64_t limbs_words = std::min(b->shape_off, b->out_words);
  // Pieces of at least 16 MiB (the copy runs at about 190 GB/s, and each piece
  // wakes the host threads once), cut between pairs.
  const int64_t piece = std::max<int64_t>((int64_t)1 << 22, limbs_words / 8 + 1);
  std::vector<int64_t> ends;  // word offsets
  std::vector<int> pair_end;  // pairs complete at each end
  for (int i = 0; i < n; ++i) {
    const int d = b->dev_index[i];
    if (d < 0) continue;
    const int64_t e = b->descs[d].out_off + (int64_t)b->plans[i].N * b->plans[i].Lout;
    if (e - (ends.empty() ? 0 : ends.back()) >= piece) {
      ends.push_back(e);
      pair_end.push_back(i + 1);
    }
  }
  if (ends.empty() || ends.back() < limbs_words) {
    ends.push_back(limbs_words);
    pair_end.push_back(n);
  }
  pair_end.back() = n;
  const int np = (int)ends.size();
  while (np > 1 && (int)b->cev.size() < np) {
    cudaEvent_t ev = nullptr;
    RS_CUDA(ctx, cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
    b->cev.push_back(ev);
  }
  cudaError_t e = cudaSuccess;
  if (np == 1 && b->out_words)  // small results: everything in one copy
    e = cudaMemcpyAsync(b->h_out, b->d_out, b->out_words * 4, cudaMemcpyDeviceToHost, b->stream);
  if (np > 1 && b->out_words > limbs_words)
    e = cudaMemcpyAsync(b->h_out + limbs_words, b->d_out + limbs_words, (b->out_words - limbs_words) * 4,
                        cudaMemcpyDeviceToHost, b->stream);
  for (int c = 0; c < np && np > 1 && e == cudaSuccess; ++c) {
    const int64_t at = c ? ends[c - 1] : 0;
    if (ends[c] > at)
      e = cudaMemcpyAsync(b->h_out + at, b->d_out + at, (ends[c] - at) * 4, cudaMemcpyDeviceToHost, b->stream);
    if (e == cudaSuccess) e = cudaEventRecord(b->cev[c], b->stream);
  }
  std::vector<int> rcs(n, RS_OK);
  struct Rows {  // rows [j0, j1) of pair i
    int i, j0, j1;
  };
  std::vector<Rows> rows;
  for (int c = 0; c < np && e == cudaSuccess; ++c) {
    e = np > 1 ? cudaEventSynchronize(b->cev[c]) : cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) break;
    if (c == 0 && device_status(b) != RS_OK) {
      cudaStreamSynchronize(b->stream);  // the other pieces still arrive in the staging buffer
      for (int i = 0; i < n && status; ++i) status[i] = RS_ERR_TIMEOUT;
      return rs_fail(ctx, RS_ERR_TIMEOUT, "tensor-core kernels: a bounded device wait ran out");
    }
    rows.clear();
    int64_t words = 0;
    for (int i = c ? pair_end[c - 1] : 0; i < pair_end[c]; ++i) {
      rcs[i] = shape_pair(b, i, out[i]);
      if (rcs[i] != RS_OK || out[i].deg < 0) continue;
      const int R = out[i].deg + 1, L = out[i].limbs;
      const int per = std::max(1, (1 << 16) / L);  // 256 KiB a task
      for (int j = 0; j < R; j += per) rows.push_back(Rows{i, j, std::min(R, j + per)});
      words += (int64_t)R * L;
    }
    // a task of a few small pairs, or of one run of rows; a thread per 128 KiB
    const int step = std::max<int>(1, (int)(rows.size() / 64));
    ctx->pool.run(((int)rows.size() + step - 1) / step, (int)std::min<int64_t>(16, words >> 15), [&](int t) {
      for (int k = t * step; k < std::min((int)rows.size(), (t + 1) * step); ++k) {
        const Rows &r = rows[k];
        const rs_upoly &o = out[r.i];
        const int Lout = b->plans[r.i].Lout, L = o.limbs;
        const uint32_t *w = b->h_out + b->descs[b->dev_index[r.i]].out_off;
        if (L == Lout) {
          memcpy(o.coeffs + (size_t)r.j0 * L, w + (size_t)r.j0 * L, (size_t)(r.j1 - r.j0) * L * 4);
        } else {
          for (int j = r.j0; j < r.j1; ++j) memcpy(o.coeffs + (size_t)j * L, w + (size_t)j * Lout, (size_t)L * 4);
        }
      }
    });
  }
  if (e != cudaSuccess) {
    cudaStreamSynchronize(b->stream);
    return rs_fail(ctx, rs_cuda_code(e), std::string("result copy: ") + cudaGetErrorString(e));
  }
  int first = RS_OK;
  for (int i = 0; i < n; ++i) {
    const int rc = rcs[i];
    if (status) status[i] = rc;
    if (rc != RS_OK && first == RS_OK) {
      first = rc;
      rs_fail(ctx, rc, std::string("pair ") + std::to_string(i) + ": " + rs_error_string(rc));
    }
  }
  return first;
}

static RsBatchOpts default_opts(rs_ctx *ctx) {
  RsBatchOpts o;
  o.use_graph = ctx->cfg.use_graphs != 0;
  o.persistent = ctx->cfg.persistent != 0;
  return o;
}

// ------------------------------------------------------------------ C ABI

extern "C" {

const char *rs_error_string(int code) {
  switch (code) {
    case RS_OK: return "ok";
    case RS_PENDING: return "pending";
    case RS_ERR_ARG: return "invalid argument";
    case RS_ERR_CAPACITY: return "output capacity too small";
    case RS_ERR_NOMEM: return "out of memory";
    case RS_ERR_CUDA: return "CUDA error";
    case RS_ERR_TIMEOUT: return "wait timed out";
    case RS_ERR_LIMIT: return "input exceeds a library limit";
    case RS_ERR_STATE: return "invalid state";
    default: return "unknown error";
  }
}

const char *rs_last_error(const rs_ctx *ctx) { return ctx ? ctx->err.c_str() : g_err.c_str(); }

int rs_test_stall_tensor_cores(rs_ctx *ctx, int32_t on) {
  if (!ctx) return rs_fail(nullptr, RS_ERR_ARG, "ctx is NULL");
  DevGuard dg(ctx->device);
  const int32_t v = on ? 1 : 0;
  RS_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  RS_CUDA(ctx, cudaMemcpy(ctx->d_stall, &v, sizeof(v), cudaMemcpyHostToDevice));
  return RS_OK;
}

int rs_config_default(rs_config *cfg) {
  if (!cfg) return rs_fail(nullptr, RS_ERR_ARG, "cfg is NULL");
  memset(cfg, 0, sizeof(*cfg));
  cfg->device = -1;
  cfg->use_graphs = 1;
  cfg->persistent = 1;
  cfg->autotune = 1;
  return RS_OK;
}

int rs_create(rs_ctx **out, const rs_config *cfg) {
  if (!out) return rs_fail(nullptr, RS_ERR_ARG, "ctx is NULL");
  *out = nullptr;
  rs_config c;
  if (cfg)
    c = *cfg;
  else
    rs_config_default(&c);
  if (c.tile_points != 0 && c.tile_points != 32 && c.tile_points != 64 && c.tile_points != 128)
    return rs_fail(nullptr, RS_ERR_ARG, "tile_points must be 0, 32, 64 or 128");
  if (c.g2_form < 0 || c.g2_form > 4) return rs_fail(nullptr, RS_ERR_ARG, "g2_form must be 0, 1, 2, 3 or 4");
  if (c.univariate < 0 || c.univariate > 1) return rs_fail(nullptr, RS_ERR_ARG, "univariate must be 0 or 1");
  if (c.crt_form < 0 || c.crt_form > 2) return rs_fail(nullptr, RS_ERR_ARG, "crt_form must be 0, 1 or 2");
  int dev = c.device;
  int ndev = 0;
  cudaError_t e = cudaGetDeviceCount(&ndev);
  if (e != cudaSuccess || ndev == 0)
    return rs_fail(nullptr, RS_ERR_CUDA, std::string("no CUDA device: ") + cudaGetErrorString(e));
  if (dev < 0 && cudaGetDevice(&dev) != cudaSuccess) dev = 0;
  if (dev >= ndev) return rs_fail(nullptr, RS_ERR_ARG, "device ordinal out of range");
  if (c.autotune_cache && c.autotune_cache[0]) {
    FILE *probe = fopen(c.autotune_cache, "r");
    if (probe) {
      fclose(probe);
      int rc0 = rs_autotune_load(c.autotune_cache);
      if (rc0 != RS_OK) return rc0;
    }
  }
  rs_ctx *ctx = new rs_ctx();
  ctx->device = dev;
  ctx->cfg = c;
  if (c.autotune_cache) ctx->tune_path = c.autotune_cache;
  ctx->cfg.autotune_cache = nullptr;  // the copy in tune_path is the one kept
  DevGuard dg(dev);
  int rc = RS_OK;
  auto chk = [&](cudaError_t e2, const char *what) {
    if (rc == RS_OK && e2 != cudaSuccess)
      rc = rs_fail(nullptr, rs_cuda_code(e2), std::string(what) + ": " + cudaGetErrorString(e2));
  };
  chk(cudaDeviceGetAttribute(&ctx->sms, cudaDevAttrMultiProcessorCount, dev), "device query");
  chk(cudaStreamCreateWithFlags(&ctx->stream, cudaStreamNonBlocking), "cudaStreamCreate");
  for (auto &ss : ctx->side) chk(cudaStreamCreateWithFlags(&ss, cudaStreamNonBlocking), "cudaStreamCreate");
  ctx->primes = rs_prime_table(RS_MAX_PRIMES);
  for (uint32_t p : ctx->primes) ctx->log2p.push_back(log2((double)p) - 1e-12);
  const int np = (int)ctx->primes.size();
  chk(cudaMalloc(&ctx->d_primes, np * 4), "cudaMalloc");
  chk(cudaMalloc(&ctx->d_mods, np * sizeof(ModP)), "cudaMalloc");
  chk(cudaMalloc(&ctx->d_vtab, (size_t)np * RS_VT_STRIDE * 4), "cudaMalloc");
  chk(cudaMalloc(&ctx->d_crt, np * 4), "cudaMalloc");
  chk(cudaMalloc(&ctx->d_qbase, np * 4), "cudaMalloc");
  chk(cudaMalloc(&ctx->d_stall, sizeof(int32_t)), "cudaMalloc");
  if (rc == RS_OK) chk(cudaMemset(ctx->d_stall, 0, sizeof(int32_t)), "cudaMemset");
  if (rc == RS_OK) chk(cudaMemcpy(ctx->d_primes, ctx->primes.data(), np * 4, cudaMemcpyHostToDevice), "cudaMemcpy");
  if (rc == RS_OK)
    chk(launch_init_primes(ctx->d_primes, np, ctx->d_mods, ctx->d_vtab, ctx->d_crt, ctx->d_qbase, ctx->stream),
        "prime tables");
  if (rc == RS_OK) {
    std::vector<uint2> tw;
    ntt_host_tables(ctx->nttc, tw);
    chk(cudaMalloc(&ctx->d_ntt_tw, tw.size() * sizeof(uint2)), "cudaMalloc");
    if (rc == RS_OK) chk(cudaMemcpy(ctx->d_ntt_tw, tw.data(), tw.size() * sizeof(uint2), cudaMemcpyHostToDevice), "cudaMemcpy");
  }
  if (rc == RS_OK) chk(cudaStreamSynchronize(ctx->stream), "prime tables");
  if (rc != RS_OK) {
    rs_destroy(ctx);
    return rc;
  }
  *out = ctx;
  return RS_OK;
}

int rs_destroy(rs_ctx *ctx) {
  if (!ctx) return RS_OK;
  rs_server_shutdown(ctx);
  if (!ctx->tune_path.empty()) rs_autotune_save(ctx->tune_path.c_str());
  {
    DevGuard dg(ctx->device);
    for (rs_batch *b : ctx->batches) rs_free_batch(b);
    if (ctx->cache) rs_free_batch(ctx->cache);
    if (ctx->sqf_cache) rs_free_batch(ctx->sqf_cache);
    if (ctx->sqf_arena) cudaFree(ctx->sqf_arena);
    if (ctx->stream) cudaStreamSynchronize(ctx->stream);
    free_tables(ctx->tab);
    for (auto &t : ctx->retired) free_tables(t);
    for (uint32_t *bh : ctx->bhat)
      if (bh) cudaFree(bh);
    for (void *bh : ctx->bhat_retired) cudaFree(bh);
    if (ctx->g2t_bt) cudaFree(ctx->g2t_bt);
    for (void *bt : ctx->g2t_retired) cudaFree(bt);
    if (ctx->g3m_wt) cudaFree(ctx->g3m_wt);
    if (ctx->g3m_rt) cudaFree(ctx->g3m_rt);
    if (ctx->g3l_bt) cudaFree(ctx->g3l_bt);
    if (ctx->g3l_cbase) cudaFree(ctx->g3l_cbase);
    for (void *wt : ctx->g3m_retired) cudaFree(wt);
    void *dev[] = {ctx->d_primes, ctx->d_mods, ctx->d_vtab, ctx->d_crt, ctx->d_qbase, ctx->d_ntt_tw, ctx->d_stall};
    for (void *p : dev)
      if (p) cudaFree(p);
    for (auto ss : ctx->side)
      if (ss) {
        cudaStreamSynchronize(ss);
        cudaStreamDestroy(ss);
      }
    if (ctx->stream) cudaStreamDestroy(ctx->stream);
  }
  delete ctx;
  return RS_OK;
}

int rs_stream(rs_ctx *ctx, void **stream) {
  if (!ctx || !stream) return rs_fail(ctx, RS_ERR_ARG, "NULL argument");
  *stream = (void *)ctx->stream;
  return RS_OK;
}

int rs_result_bound(const rs_bipoly *f, const rs_bipoly *g, int32_t *deg_bound, int32_t *limbs_bound,
                    int32_t *primes, int32_t *bits) {
  static const std::vector<double> log2p = [] {
    std::vector<double> v;
    for (uint32_t p : rs_prime_table(RS_MAX_PRIMES)) v.push_back(log2((double)p) - 1e-12);
    return v;
  }();
  PairPlan p;
  const char *why = "";
  int rc = rs_plan_pair(f, g, log2p, p, &why);
  if (rc != RS_OK) return rs_fail(nullptr, rc, why);
  if (deg_bound) *deg_bound = p.trivial_zero ? -1 : p.D;
  if (limbs_bound) *limbs_bound = p.Lout;
  if (primes) *primes = p.K;
  if (bits) *bits = p.bits;
  return RS_OK;
}

int rs_batch_create_on(rs_ctx *ctx, int32_t n, const rs_bipoly *f, const rs_bipoly *g, void *stream,
                       rs_batch **batch) {
  if (!ctx || !batch || n < 0 || (n > 0 && (!f || !g))) return rs_fail(ctx, RS_ERR_ARG, "NULL argument or negative n");
  *batch = nullptr;
  std::vector<PairPlan> plans;
  int first = RS_OK;
  rs_plan_all(ctx, n, f, g, plans, nullptr, &first);
  rs_batch *b = nullptr;
  RsBatchOpts o = default_opts(ctx);
  o.stream = static_cast<cudaStream_t>(stream);
  int rc = rs_build_batch(ctx, n, f, g, std::move(plans), o, &b);
  if (rc != RS_OK) return rc;
  DevGuard dg(ctx->device);
  rc = rs_upload(b, f, g);
  if (rc != RS_OK) {
    rs_free_batch(b);
    return rc;
  }
  ctx->batches.push_back(b);
  *batch = b;
  return RS_OK;
}

int rs_batch_create(rs_ctx *ctx, int32_t n, const rs_bipoly *f, const rs_bipoly *g, rs_batch **batch) {
  return rs_batch_create_on(ctx, n, f, g, nullptr, batch);
}

int rs_batch_upload(rs_batch *b, int32_t n, const rs_bipoly *f, const rs_bipoly *g) {
  if (!b || n != b->n || (n > 0 && (!f || !g))) return rs_fail(b ? b->ctx : nullptr, RS_ERR_ARG, "bad arguments");
  // Each pair is planned and compared by one task, which frees the plan again.
  std::vector<char> same(n, 0);
  int step = 1;
  const int threads = plan_threads(n, f, g, &step);
  b->ctx->pool.run((n + step - 1) / step, threads, [&](int t) {
    for (int i = t * step; i < std::min(n, (t + 1) * step); ++i) {
      PairPlan plan;
      const char *why = "";
      plan_one(b->ctx, f[i], g[i], plan, &why);
      same[i] = rs_same_shape(plan, b->plans[i]);
    }
  });
  for (int i = 0; i < n; ++i)
    if (!same[i])
      return rs_fail(b->ctx, RS_ERR_STATE, "inputs do not match the batch's plan (pair " + std::to_string(i) + ")");
  DevGuard dg(b->ctx->device);
  return rs_upload(b, f, g);
}

int rs_batch_run(rs_batch *b) {
  if (!b) return rs_fail(nullptr, RS_ERR_ARG, "batch is NULL");
  return rs_run(b);
}

int rs_batch_sync(rs_batch *b) {
  if (!b) return rs_fail(nullptr, RS_ERR_ARG, "batch is NULL");
  DevGuard dg(b->ctx->device);
  RS_CUDA(b->ctx, cudaStreamSynchronize(b->stream));
  return RS_OK;
}

int rs_batch_results(rs_batch *b, rs_upoly *out, int32_t *status) {
  if (!b || (b->n > 0 && !out)) return rs_fail(b ? b->ctx : nullptr, RS_ERR_ARG, "NULL argument");
  return fetch(b, out, status);
}

int rs_batch_destroy(rs_batch *b) {
  if (!b) return RS_OK;
  auto &v = b->ctx->batches;
  v.erase(std::remove(v.begin(), v.end(), b), v.end());
  rs_free_batch(b);
  return RS_OK;
}

int rs_batch_info_get(rs_batch *b, rs_batch_info *info) {
  if (!b || !info) return rs_fail(b ? b->ctx : nullptr, RS_ERR_ARG, "NULL argument");
  rs_ctx *ctx = b->ctx;
  DevGuard dg(ctx->device);
  *info = b->info;
  info->ms_images = info->ms_interp = info->ms_crt = info->ms_total = -1.0f;
  info->ms_yun = 0.0f;
  info->reserved = 0;
  if (!b->ran) return RS_OK;
  RS_CUDA(ctx, cudaStreamSynchronize(b->stream));
  unsigned long long st[ST_COUNT];
  RS_CUDA(ctx, cudaMemcpy(st, b->d_stats, sizeof(st), cudaMemcpyDeviceToHost));
  info->unlucky_points = (int64_t)st[ST_UNLUCKY_POINTS];
  info->degenerate_images = (int64_t)st[ST_DEGENERATE];
  info->unlucky_primes = (int64_t)st[ST_UNLUCKY_PRIMES];
  if (ctx->cfg.timing) {
    float t = 0;
    if (cudaEventElapsedTime(&t, b->ev[0], b->ev[1]) == cudaSuccess) info->ms_images = t;
    if (!b->opt.images_only) {
      if (cudaEventElapsedTime(&t, b->ev[1], b->ev[b->nyun ? 4 : 2]) == cudaSuccess) info->ms_interp = t;
      if (b->nyun && cudaEventElapsedTime(&t, b->ev[4], b->ev[2]) == cudaSuccess) info->ms_yun = t;
      if (cudaEventElapsedTime(&t, b->ev[2], b->ev[3]) == cudaSuccess) info->ms_crt = t;
      if (cudaEventElapsedTime(&t, b->ev[0], b->ev[3]) == cudaSuccess) info->ms_total = t;
    }
  }
  return RS_OK;
}

int rs_resultant_batch(rs_ctx *ctx, int32_t n, const rs_bipoly *f, const rs_bipoly *g, rs_upoly *out,
                       int32_t *status) {
  if (!ctx || n < 0 || (n > 0 && (!f || !g || !out))) return rs_fail(ctx, RS_ERR_ARG, "NULL argument or negative n");
  if (n == 0) return RS_OK;
  std::vector<PairPlan> plans;
  int first = RS_OK;
  rs_plan_all(ctx, n, f, g, plans, status, &first);
  rs_batch *b = ctx->cache;
  bool reuse = b && b->n == n;
  for (int i = 0; reuse && i < n; ++i) reuse = rs_same_shape(plans[i], b->plans[i]);
  if (!reuse) {
    if (b) rs_free_batch(b);
    ctx->cache = nullptr;
    int rc = rs_build_batch(ctx, n, f, g, std::move(plans), default_opts(ctx), &b);
    if (rc != RS_OK) return rc;
    ctx->cache = b;
  }
  DevGuard dg(ctx->device);
  int rc = rs_upload(b, f, g);
  if (rc == RS_OK) rc = rs_run(b);
  if (rc == RS_OK) rc = fetch(b, out, status);
  return rc != RS_OK ? rc : first;
}

int rs_resultant_y(rs_ctx *ctx, const rs_bipoly *f, const rs_bipoly *g, rs_upoly *out) {
  return rs_resultant_batch(ctx, 1, f, g, out, nullptr);
}

// Copy of p with x and y exchanged (storage in `buf`); an input the planner
// would reject is passed through unchanged so that it fails the same way.
static rs_bipoly transposed(const rs_bipoly &p, std::vector<uint32_t> &buf) {
  if (!p.coeffs || p.deg_x < 0 || p.deg_y < 0 || p.limbs < 1 || p.limbs > RS_MAX_LIMBS ||
      ((int64_t)p.deg_x + 1) * ((int64_t)p.deg_y + 1) > ((int64_t)1 << 26))
    return p;
  const int nx = p.deg_x + 1, ny = p.deg_y + 1, L = p.limbs;
  buf.resize((size_t)nx * ny * L);
  for (int i = 0; i < nx; ++i)
    for (int j = 0; j < ny; ++j)
      memcpy(&buf[((size_t)j * nx + i) * L], p.coeffs + ((size_t)i * ny + j) * L, (size_t)L * 4);
  rs_bipoly t;
  t.deg_x = p.deg_y;
  t.deg_y = p.deg_x;
  t.limbs = L;
  t.coeffs = buf.data();
  return t;
}

int rs_resultant_x(rs_ctx *ctx, const rs_bipoly *f, const rs_bipoly *g, rs_upoly *out) {
  if (!ctx || !f || !g || !out) return rs_fail(ctx, RS_ERR_ARG, "NULL argument");
  std::vector<uint32_t> bf, bg;
  const rs_bipoly ft = transposed(*f, bf), gt = transposed(*g, bg);
  return rs_resultant_batch(ctx, 1, &ft, &gt, out, nullptr);
}

int rs_squarefree_projections(rs_ctx *ctx, int32_t n, const rs_bipoly *f, const rs_bipoly *g, int32_t max_mult,
                              rs_upoly *content_y, rs_upoly *factors_y, int32_t *nmult_y, rs_upoly *content_x,
                              rs_upoly *factors_x, int32_t *nmult_x, int32_t *status) {
  if (!ctx || n < 0 || max_mult < 1 ||
      (n > 0 && (!f || !g || !content_y || !factors_y || !nmult_y || !content_x || !factors_x || !nmult_x)))
    return rs_fail(ctx, RS_ERR_ARG, "NULL argument, negative n or max_mult < 1");
  if (n == 0) return RS_OK;
  const size_t N2 = 2 * (size_t)n, M = (size_t)max_mult;
  std::vector<std::vector<uint32_t>> bufs(N2);
  std::vector<rs_bipoly> F(N2), G(N2);
  std::vector<rs_upoly> C(N2), FA(N2 * M);
  std::vector<int32_t> NM(N2, 0);
  for (int i = 0; i < n; ++i) {
    F[i] = f[i];
    G[i] = g[i];
    F[n + i] = transposed(f[i], bufs[2 * (size_t)i]);
    G[n + i] = transposed(g[i], bufs[2 * (size_t)i + 1]);
    C[i] = content_y[i];
    C[n + i] = content_x[i];
    for (size_t m = 0; m < M; ++m) {
      FA[i * M + m] = factors_y[i * M + m];
      FA[(n + i) * M + m] = factors_x[i * M + m];
    }
  }
  const int rc = rs_squarefree_batch(ctx, 2 * n, F.data(), G.data(), max_mult, C.data(), FA.data(), NM.data(),
                                     status);
  for (int i = 0; i < n; ++i) {  // shapes (and data, through the caller's pointers) back
    content_y[i] = C[i];
    content_x[i] = C[n + i];
    nmult_y[i] = NM[i];
    nmult_x[i] = NM[n + i];
    for (size_t m = 0; m < M; ++m) {
      factors_y[i * M + m] = FA[i * M + m];
      factors_x[i * M + m] = FA[(n + i) * M + m];
    }
  }
  return rc;
}

int rs_projections(rs_ctx *ctx, int32_t n, const rs_bipoly *f, const rs_bipoly *g, rs_upoly *out_y,
                   rs_upoly *out_x, int32_t *status) {
  if (!ctx || n < 0 || (n > 0 && (!f || !g || !out_y || !out_x)))
    return rs_fail(ctx, RS_ERR_ARG, "NULL argument or negative n");
  if (n == 0) return RS_OK;
  std::vector<std::vector<uint32_t>> bufs(2 * (size_t)n);
  std::vector<rs_bipoly> F(2 * (size_t)n), G(2 * (size_t)n);
  std::vector<rs_upoly> O(2 * (size_t)n);
  for (int i = 0; i < n; ++i) {
    F[i] = f[i];
    G[i] = g[i];
    F[n + i] = transposed(f[i], bufs[2 * (size_t)i]);
    G[n + i] = transposed(g[i], bufs[2 * (size_t)i + 1]);
    O[i] = out_y[i];
    O[n + i] = out_x[i];
  }
  const int rc = rs_resultant_batch(ctx, 2 * n, F.data(), G.data(), O.data(), status);
  for (int i = 0; i < n; ++i) {  // deg and limbs are written on success and on RS_ERR_CAPACITY
    out_y[i].deg = O[i].deg;
    out_y[i].limbs = O[i].limbs;
    out_x[i].deg = O[n + i].deg;
    out_x[i].limbs = O[n + i].limbs;
  }
  return rc;
}

int rs_images(rs_ctx *ctx, const rs_bipoly *f, const rs_bipoly *g, int32_t nprimes, int32_t npoints,
              uint32_t *primes_out, uint32_t *points_out, uint32_t *images_out) {
  if (!ctx || !f || !g || !images_out || nprimes < 1 || npoints < 1)
    return rs_fail(ctx, RS_ERR_ARG, "bad arguments");
  if (nprimes > (int)ctx->primes.size() || npoints > RS_MAX_POINTS)
    return rs_fail(ctx, RS_ERR_LIMIT, "nprimes or npoints above the library limits");
  std::vector<PairPlan> plans;
  int first = RS_OK;
  rs_plan_all(ctx, 1, f, g, plans, nullptr, &first);
  if (first != RS_OK) return first;
  DevGuard dg(ctx->device);
  if (plans[0].trivial_zero) {
    memset(images_out, 0, (size_t)nprimes * npoints * 4);
    if (points_out) {
      std::vector<uint32_t> qb(nprimes);
      RS_CUDA(ctx, cudaMemcpy(qb.data(), ctx->d_qbase, (size_t)nprimes * 4, cudaMemcpyDeviceToHost));
      for (int k = 0; k < nprimes; ++k) {
        const ModP m = make_modp(ctx->primes[k]);
        for (int i = 0; i < npoints; ++i) {  // point 2 t + s is (-1)^s q^t
          const uint32_t pw = from_mont(mpow(qb[k], (uint32_t)(i >> 1), m), m);
          points_out[(size_t)k * npoints + i] = (i & 1) ? mneg(pw, m.p) : pw;
        }
      }
    }
  } else {
    plans[0].K = nprimes;
    plans[0].N = npoints;
    plans[0].D = npoints - 1;
    plans[0].Lout = 1;
    plans[0].cap = std::max(plans[0].f.my, plans[0].g.my) + 1;
    RsBatchOpts o = default_opts(ctx);
    o.images_only = true;
    o.use_graph = false;
    o.tune = false;
    rs_batch *b = nullptr;
    int rc = rs_build_batch(ctx, 1, f, g, std::move(plans), o, &b);
    if (rc != RS_OK) return rc;
    rc = rs_upload(b, f, g);
    if (rc == RS_OK) rc = rs_run(b);
    if (rc == RS_OK) {
      uint32_t *d_pts = points_out ? b->d_out : nullptr;  // images-only batches size d_out to K * N
      cudaError_t e = launch_finalize_images(ctx->d_mods, ctx->d_qbase, b->d_num, b->d_den, b->d_xl, d_pts,
                                             nprimes, npoints, b->descs[0].NI, b->stream);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(images_out, b->d_xl, (size_t)nprimes * npoints * 4, cudaMemcpyDeviceToHost, b->stream);
      if (e == cudaSuccess && points_out)
        e = cudaMemcpyAsync(points_out, d_pts, (size_t)nprimes * npoints * 4, cudaMemcpyDeviceToHost, b->stream);
      if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
      if (e != cudaSuccess) rc = rs_fail(ctx, RS_ERR_CUDA, std::string("images: ") + cudaGetErrorString(e));
    }
    rs_free_batch(b);
    if (rc != RS_OK) return rc;
  }
  if (primes_out) memcpy(primes_out, ctx->primes.data(), (size_t)nprimes * 4);
  return RS_OK;
}

}  // extern "C"
