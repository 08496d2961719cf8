// G2 (interpolation mod p) and the per-prime constant tables.  Paper,
// Section 4.1: R^{(y)} is interpolated over Z_p from the images z_i^{(p)}
// (a Vandermonde solve); the Chinese remaindering is in kernels_g3.cu.
#include "../../include/rs.h"
#include "blockinv.cuh"
#include "rs_internal.cuh"

namespace {

// Interpolation at the geometric points x_i = q^i, i = 0..D (Section 4.1
// asks for the Vandermonde solve; on a geometric progression it factors into
// two convolutions).  With F_t = prod_{s=1}^t (q^s - 1) and
// b_t = (-1)^t q^{C(t,2)} / F_t:
//   Newton coefficients  c_k = q^{-C(k,2)} sum_{j<=k} (z_j / F_j) b_{k-j}
//   (the divided differences on a geometric progression, since
//   prod_{l<=k, l!=j} (q^j - q^l) = q^{C(k,2)} (-1)^{k-j} F_j F_{k-j} / q^{C(k-j,2)}),
//   monomial coefficients R_m = (1 / F_m) sum_{t<=D-m} (c_{m+t} F_{m+t}) b_t
//   (q-binomial expansion of prod_{j<k} (x - q^j)).
// Both sums are the convolution conv(x, b)_k = sum_{j<=k} x_j b_{k-j}, the
// second one on the reversed sequence.  Residues enter it as signed
// representatives |v| < 2^30, so 7 products accumulate exactly in an int64
// and one fold S = hi 2^32 + lo -> hi (2^32 mod p) + lo keeps |S| < 2^53
// (every table prime exceeds 2^31 - 2^20, so 2^32 mod p <= 2^21).


__device__ __forceinline__ int32_t signed_rep(uint32_t v, uint32_t p) {
  return v > (p >> 1) ? (int32_t)v - (int32_t)p : (int32_t)v;
}

// Reduce a folded accumulator, or the difference of two (|s| < 2^54), to
// [0, p), divided by 2^32.
__device__ __forceinline__ uint32_t finish64(int64_t s, const ModP &m) {
  const uint64_t t = (uint64_t)(s + ((int64_t)m.p << 24));  // 0 <= t < 2^56 < p 2^32
  return redc(t, m.p, m.pinv);
}

// The direct convolution's work, split over a block.  Outputs come in blocks
// of R; output block bi needs bi + 1 chunks of R inputs, so the pair of blocks
// (pi, nblk - 1 - pi) needs nblk + 1 chunks for every pi.  That walk of
// nblk + 1 chunks is cut into S segments of `len` chunks; each segment writes
// its partial sums of both blocks, reduced to [0, p), and conv_value adds them.
struct ConvShape {
  int n, S, nblk, npair, len;
};

__device__ __forceinline__ ConvShape conv_shape(int n, int S) {
  ConvShape c;
  c.n = n;
  c.S = S;
  c.nblk = (n + RS_CONV_R - 1) / RS_CONV_R;
  c.npair = (c.nblk + 1) / 2;
  c.len = (c.nblk + S) / S;  // ceil((nblk + 1) / S)
  return c;
}

// Partial sums of sum_{j<=k} x[j] b[k-j], k < n, of `nh` inputs x, x + W
// against one b: part[(h S + s) n + k] over segment s of input h.  x and b
// hold signed representatives and are zero for indices in [-RS_G2_PAD, 0) and
// [n, n + RS_G2_PAD).
//
// Neighbouring lanes take neighbouring block pairs of one segment.  While both
// walk their low block they read b words R apart (R odd: distinct banks) and
// the same x words, in the mirror blocks the same b words and x words R apart;
// every unit of a segment has the same trip count.  Lanes leave their low
// block in different steps, so a step only keeps the sums of that moment
// (snap) and the mirror block's are the difference at the end.
__device__ void conv_parts(const int32_t *x, const int32_t *b, uint32_t *part, const ConvShape &cs, int nh, int W,
                           const ModP &m) {
  constexpr int R = RS_CONV_R;
  const int n = cs.n, units = nh * cs.S * cs.npair;
  for (int u = threadIdx.x; u < units; u += blockDim.x) {
    const int hs = u / cs.npair, pi = u - hs * cs.npair;
    const int h = hs >= cs.S, s = hs - h * cs.S;
    const int hb = cs.nblk - 1 - pi;
    const int c0 = s * cs.len;
    const int steps = min(cs.len, (hb == pi ? pi + 1 : cs.nblk + 1) - c0);  // the middle block once
    const bool low = c0 <= pi;
    const int turn = low ? pi - c0 : -1;  // step that completes the low block
    const int32_t *xp = x + h * W + (low ? c0 : c0 - pi - 1) * R;
    const int32_t *bp = b + ((low ? pi - c0 : hb - (c0 - pi - 1)) * R - (R - 1));
    int64_t acc[R], snap[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = snap[r] = 0;
#pragma unroll 1
    for (int c = 0; c < steps; ++c) {
      int32_t bw[2 * R - 1], av[R];
#pragma unroll
      for (int i = 0; i < 2 * R - 1; ++i) bw[i] = bp[i];
#pragma unroll
      for (int i = 0; i < R; ++i) av[i] = xp[i];
      xp += R;
      bp -= R;
#pragma unroll
      for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int jj = 0; jj < R; ++jj) acc[r] = rs_mac_s32(acc[r], av[jj], bw[(R - 1) + r - jj]);
        acc[r] = rs_fold64(acc[r], m.r1);
      }
      if (c == turn) {  // on to the mirror block
#pragma unroll
        for (int r = 0; r < R; ++r) snap[r] = acc[r];
        xp = x + h * W;
        bp = b + (hb * R - (R - 1));
      }
    }
    const bool kept = steps <= turn;  // the segment ends in the low block
    uint32_t *y = part + (size_t)hs * n;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int64_t lo = kept ? acc[r] : snap[r];
      if (pi * R + r < n) y[pi * R + r] = finish64(lo, m);
      if (hb != pi && hb * R + r < n) y[hb * R + r] = finish64(acc[r] - lo, m);
    }
  }
}

// Sum of the segments' partial sums of output k of input h.
__device__ __forceinline__ uint32_t conv_value(const uint32_t *part, const ConvShape &cs, int h, int k, const ModP &m) {
  const uint32_t *y = part + (size_t)h * cs.S * cs.n + k;
  uint32_t v = y[0];
  for (int s = 1; s < cs.S; ++s) {
    y += cs.n;
    v = madd(v, y[0], m.p);
  }
  return v;
}

// Cluster barrier of a pair of blocks, in two halves.
__device__ __forceinline__ void pair_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void pair_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// One block, or a cluster of two, per (pair, prime).  The images come in pairs
// z+-_i at +-q^i, i < M = NI / 2, with R(x) = E(x^2) + x O(x^2):
//   E(Q^i) = (z+_i + z-_i) / 2,  O(Q^i) = (z+_i - z-_i) / (2 q^i),  Q = q^2,
// and with z = num / den both are fractions over D_i = den+ den-, inverted
// together.  E and O (degrees < M) are then interpolated on the geometric
// points Q^i by the two convolutions above, giving the even and the odd
// coefficients of R: both at once (a.halves = 2), in turn (1), or one in each
// block of a cluster (a.split).  The residues may replace the numerators, so
// in a cluster neither block writes before both have read.  Shared memory:
// inputs of E and O and b, each of M words with RS_G2_PAD zero words on both
// sides, and the partial sums (g2_seg segments of M words per half at once;
// the inverses before that).
//
// Bound by the multiplier pipe (73% busy at 10,280 tasks of M = 113: a third
// of it the convolutions' wide products, the rest modular products of the
// steps around them), and for few tasks by a block's latency.  With one thread
// per block pair and the halves in turn 3 to 33 lanes of a block worked;
// splitting the walks fills them.  G2 stage, us, before (the fastest of the
// three forms) -> now: 69 tasks of M = 451: 70 -> 18; 8,844 of 5 to 61: 83 ->
// 36; 23,980 of 41: 248 -> 96; 10,280 of 113: 236 -> 117; 40,000 of 113: 860 ->
// 422; 546 of 2,049: 880 -> 853; 1,127 of 169 to 1,369: 380 -> 266.  Of these a
// thread's first point's loads taken together at the start gave 20.4 -> 18.2
// with 69 tasks and about 1% with 10,280 and more.
__global__ void __launch_bounds__(512, 2) g2_kernel(G2Args a) {
  extern __shared__ __align__(16) uint32_t sm[];
  __shared__ uint32_t scratch[128];
  const int split = a.split;
  const int2 task = a.tasks[blockIdx.x >> split];
  const PairDesc pd = a.pairs[task.x];
  const ModP m = a.mods[task.y];
  const int N = pd.N, NI = pd.NI, M = NI >> 1, D = M - 1, T = blockDim.x, tid = threadIdx.x;
  const int W = M + 2 * RS_G2_PAD;
  const int nh = split ? 1 : 2, h0 = split ? (blockIdx.x & 1) : 0;  // halves of this block
  const int hc = a.halves;                                         // of those, at once
  int32_t *X = reinterpret_cast<int32_t *>(sm) + RS_G2_PAD;
  int32_t *Bs = X + nh * W;
  uint32_t *Y = reinterpret_cast<uint32_t *>(Bs + W - RS_G2_PAD);
  const size_t base = (size_t)pd.img_off + (size_t)task.y * NI;
  const size_t tb = (size_t)task.y * a.tab_stride;
  const uint32_t *finv = a.finv + tb, *gt = a.gtab + tb, *hq = a.hq + tb;
  const int32_t *bt = a.btab + tb;

  // a thread's first point: its images and table entries, all on their way before the first is needed
  const int f = min(tid, M - 1);
  const uint32_t np0 = a.num[base + 2 * f], dp0 = a.den[base + 2 * f];
  const uint32_t nm0 = a.num[base + 2 * f + 1], dm0 = a.den[base + 2 * f + 1];
  const uint32_t fi0 = finv[f], hq0 = hq[f], hqe = hq[0], gt0 = gt[f];
  const int32_t bt0 = bt[f];
  uint32_t *dens = reinterpret_cast<uint32_t *>(Bs);
  if (tid < M) dens[tid] = mmul(dp0, dm0, m);
  for (int i = tid + T; i < M; i += T) dens[i] = mmul(a.den[base + 2 * i], a.den[base + 2 * i + 1], m);
  __syncthreads();
  batch_invert(dens, Y, M, m, scratch, true);  // plain inverses: from here on plain times Montgomery form
  __syncthreads();
  for (int i = tid; i < M; i += T) {
    const bool f0 = i < T;
    const uint32_t np = f0 ? np0 : a.num[base + 2 * i], dp = f0 ? dp0 : a.den[base + 2 * i];
    const uint32_t nm = f0 ? nm0 : a.num[base + 2 * i + 1], dm = f0 ? dm0 : a.den[base + 2 * i + 1];
    const uint32_t fy = mmul(f0 ? fi0 : finv[i], Y[i], m);
    for (int h = 0; h < nh; ++h) {
      const bool odd = (h0 + h) != 0;
      const uint32_t v = mmul2(np, dm, odd ? mneg(nm, m.p) : nm, dp, m);  // z+ +- z-
      // E / F_i or O / F_i; hq[0] = 1/2
      X[h * W + i] = signed_rep(mmul(mmul(v, odd ? (f0 ? hq0 : hq[i]) : hqe, m), fy, m), m.p);
    }
  }
  if (split) pair_arrive();
  for (int i = tid; i < M; i += T) Bs[i] = i < T ? bt0 : bt[i];
  for (int i = tid; i < RS_G2_PAD; i += T) {
    for (int h = 0; h < nh; ++h) {
      X[h * W - 1 - i] = 0;
      X[h * W + M + i] = 0;
    }
    Bs[-1 - i] = 0;
    Bs[M + i] = 0;
  }
  __syncthreads();
  const ConvShape cs = conv_shape(M, pd.g2_seg);
  for (int hh = 0; hh < nh; hh += hc) {
    int32_t *x = X + hh * W;
    conv_parts(x, Bs, Y, cs, hc, W, m);  // Y: Q^{C(k,2)} c_k
    __syncthreads();
    for (int k = tid; k < M; k += T) {
      const uint32_t g = k < T ? gt0 : gt[k];
      for (int h = 0; h < hc; ++h)
        x[h * W + D - k] = signed_rep(mmul(conv_value(Y, cs, h, k, m), g, m), m.p);  // c_k F_k reversed
    }
    __syncthreads();
    conv_parts(x, Bs, Y, cs, hc, W, m);  // Y[D - t]: sum_s c_{t+s} F_{t+s} b_s
    __syncthreads();
    if (split) pair_wait();
    for (int i = tid; i < M; i += T) {
      const uint32_t fi = i < T ? fi0 : finv[i];
      for (int h = 0; h < hc; ++h) {
        const int c = 2 * i + h0 + hh + h;
        if (c < N) a.coef[base + c] = mmul(conv_value(Y, cs, h, D - i, m), fi, m);
      }
    }
    __syncthreads();
  }
}

// Per prime k < K, with q its point base and Q = q^2: for t < stride the
// chirp tables Q^{C(t,2)} (signed representative) and Q^{-C(t,2)} and the
// powers q^t (evaluation in G1), and for t < N the interpolation tables
// 1 / F_t, Q^{-C(t,2)} F_t, the signed (-1)^t Q^{C(t,2)} / F_t,
// F_t = prod_{s=1}^t (Q^s - 1), and 1 / (2 q^t) (G2; finv may be NULL when
// only the chirp tables are wanted).  One thread per prime.
__global__ void tables_kernel(const ModP *mods, const uint32_t *qbase, int K, int N, int stride,
                              uint32_t *finv, uint32_t *gtab, int32_t *btab, uint32_t *hqt, int32_t *qct,
                              uint32_t *qnt, uint32_t *qpt) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= K) return;
  const ModP m = mods[k];
  const uint32_t qb = qbase[k], qbi = minv(qb, m);
  const uint32_t q = mmul(qb, qb, m), qi = minv(q, m);  // Q and 1/Q
  {
    // the chirp tables of the evaluation, base q: q^{C(t,2)}, q^{-C(t,2)}, and q^t
    uint32_t up = m.r1, dn = m.r1, pw = m.r1, piw = m.r1;  // q^{C(t,2)}, q^{-C(t,2)}, q^t, q^{-t}
    int32_t *qc = qct + (size_t)k * stride;
    uint32_t *qn = qnt + (size_t)k * stride;
    uint32_t *qp = qpt + (size_t)k * stride;
    for (int t = 0; t < stride; ++t) {
      qc[t] = signed_rep(up, m.p);
      qn[t] = dn;
      qp[t] = pw;
      up = mmul(up, pw, m);  // C(t+1,2) = C(t,2) + t
      dn = mmul(dn, piw, m);
      pw = mmul(pw, qb, m);
      piw = mmul(piw, qbi, m);
    }
  }
  if (!finv) return;
  uint32_t *fi = finv + (size_t)k * N, *gt = gtab + (size_t)k * N, *hq = hqt + (size_t)k * N;
  int32_t *bt = btab + (size_t)k * N;
  {
    const uint32_t inv2 = minv(madd(m.r1, m.r1, m.p), m);
    uint32_t w = inv2;  // 1 / (2 q^t)
    for (int t = 0; t < N; ++t) {
      hq[t] = w;
      w = mmul(w, qbi, m);
    }
  }
  // forward: F_t (kept in fi for now) and Q^{-C(t,2)} (kept in gt)
  uint32_t F = m.r1, qt = m.r1, qneg = m.r1, qinvt = m.r1;  // Q^t, Q^{-C(t,2)}, Q^{-(t-1)}
  for (int t = 0; t < N; ++t) {
    if (t > 0) {
      qt = mmul(qt, q, m);
      F = mmul(F, msub(qt, m.r1, m.p), m);
      if (t > 1) qinvt = mmul(qinvt, qi, m);
      qneg = mmul(qneg, qinvt, m);
    }
    fi[t] = F;
    gt[t] = qneg;
  }
  // backward: 1 / F_t from 1 / F_{N-1}; Q^{C(t,2)} from Q^{C(N-1,2)}
  uint32_t inv = minv(F, m);
  uint32_t qc = minv(qneg, m);  // Q^{C(N-1,2)}
  uint32_t qm1 = qinvt;         // Q^{-(t-1)} at t = N-1
  for (int t = N - 1; t >= 0; --t) {
    const uint32_t Ft = fi[t];
    fi[t] = inv;
    uint32_t bv = mmul(qc, inv, m);
    if (t & 1) bv = mneg(bv, m.p);
    bt[t] = signed_rep(bv, m.p);
    gt[t] = mmul(gt[t], Ft, m);
    if (t > 0) {
      inv = mmul(inv, msub(qt, m.r1, m.p), m);  // 1/F_{t-1} = (Q^t - 1) / F_t
      qt = mmul(qt, qi, m);
      qc = mmul(qc, qm1, m);                    // Q^{C(t-1,2)} = Q^{C(t,2)} Q^{-(t-1)}
      qm1 = mmul(qm1, q, m);
    }
  }
}

// Per prime: Montgomery constants, V[l] = 2^(32 l) R^2 mod p (limb weights
// for the modular reduction of input coefficients) and the Garner constant
// (p_0 ... p_{k-1})^{-1} mod p_k.
__global__ void init_primes_kernel(const uint32_t *primes, int n, ModP *mods, uint32_t *vtab,
                                   uint32_t *crt, uint32_t *qbase) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const ModP m = make_modp(primes[k]);
  mods[k] = m;
  uint32_t v = m.r2;
  for (int l = 0; l < RS_VT_STRIDE; ++l) {
    vtab[(size_t)k * RS_VT_STRIDE + l] = v;
    v = mmul(v, m.r2, m);
  }
  uint32_t acc = m.r1;
  for (int l = 0; l < k; ++l) acc = mmul(acc, to_mont(primes[l] - m.p, m), m);
  crt[k] = minv(acc, m);
  // base of the evaluation points: the smallest q >= 2 whose powers
  // q^1 .. q^RS_MAX_POINTS all differ from 1.  Then the points +-q^i,
  // i < RS_MAX_POINTS / 2, are distinct (q^d = -1 would give q^(2d) = 1 with
  // 2d <= RS_MAX_POINTS) and every Q^t - 1 = q^(2t) - 1, 0 < t <
  // RS_MAX_POINTS / 2, is invertible.
  for (uint32_t c = 2;; ++c) {
    const uint32_t qm = to_mont(c, m);
    uint32_t x = qm;
    int t = 1;
    while (t <= RS_MAX_POINTS && x != m.r1) {
      x = mmul(x, qm, m);
      ++t;
    }
    if (t > RS_MAX_POINTS) {
      qbase[k] = qm;
      break;
    }
  }
}

__global__ void finalize_images_kernel(const ModP *mods, const uint32_t *qbase, const uint32_t *num,
                                       const uint32_t *den, uint32_t *z, uint32_t *points, int K,
                                       int N, int NI) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (size_t)K * N) return;
  const int k = (int)(i / N), x = (int)(i % N);
  const ModP m = mods[k];
  const size_t src = (size_t)k * NI + x;
  z[i] = from_mont(mmul(num[src], minv(den[src], m), m), m);
  if (points) {  // image 2 i + s is at (-1)^s q^i
    const uint32_t pw = from_mont(mpow(qbase[k], (uint32_t)(x >> 1), m), m);
    points[i] = (x & 1) ? mneg(pw, m.p) : pw;
  }
}

}  // namespace

cudaError_t launch_tables(const ModP *mods, const uint32_t *qbase, int K, int N, int stride,
                          uint32_t *finv, uint32_t *gtab, int32_t *btab, uint32_t *hq, int32_t *qc,
                          uint32_t *qn, uint32_t *qp, cudaStream_t s) {
  tables_kernel<<<(K + 63) / 64, 64, 0, s>>>(mods, qbase, K, N, stride, finv, gtab, btab, hq, qc, qn, qp);
  return cudaGetLastError();
}

cudaError_t g2_prepare() {  // per-kernel attribute: allow the largest any plan may need
  cudaError_t e = cudaFuncSetAttribute(g2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, RS_G2_MAX_SMEM_BYTES);
  // one carveout for every class: launches that want different ones don't share an SM
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(g2_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  return e;
}

cudaError_t launch_g2(int threads, int blocks, size_t smem, const G2Args &a, cudaStream_t s) {
  if (!a.split) {
    g2_kernel<<<blocks, threads, smem, s>>>(a);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(2 * blocks);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, g2_kernel, a);
}


cudaError_t launch_init_primes(const uint32_t *primes, int n, ModP *mods, uint32_t *vtab,
                               uint32_t *crt, uint32_t *qbase, cudaStream_t s) {
  init_primes_kernel<<<(n + 127) / 128, 128, 0, s>>>(primes, n, mods, vtab, crt, qbase);
  return cudaGetLastError();
}

cudaError_t launch_finalize_images(const ModP *mods, const uint32_t *qbase, const uint32_t *num,
                                   const uint32_t *den, uint32_t *z, uint32_t *points, int K, int N,
                                   int NI, cudaStream_t s) {
  const size_t n = (size_t)K * N;
  finalize_images_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(mods, qbase, num, den, z, points,
                                                                      K, N, NI);
  return cudaGetLastError();
}
