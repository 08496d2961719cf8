// G3: Chinese remaindering (paper, Section 4.1: the residues R mod p are
// combined into the integer result by the Chinese remainder theorem).
//
// Garner's mixed-radix form R_j = v_0 + p_0 (v_1 + p_1 (v_2 + ...)) with
// digits v_k in the symmetric range (-p_k/2, p_k/2) gives the symmetric
// representative of R_j mod p_0 ... p_{K-1} directly.  Digit k is
//   v_k = (r_k - sum_{l<k} v_l W[k][l]) c_k  (mod p_k),
//   W[k][l] = p_0 ... p_{l-1} mod p_k,  c_k = (p_0 ... p_{k-1})^{-1} mod p_k,
// and the integer is R_j = sum_k v_k P_k with P_k = p_0 ... p_{k-1}.
//
// G3t: the digits, in tiles of 32 coefficients by blocks of 64 digits (a
//      rectangular update from the earlier digits, then a small triangular
//      solve), every dot product lazily accumulated in int64.
// G3b: one thread per (coefficient, chunk of 16 limbs of R_j) accumulates
//      sum_k w_k P_k[h] with the offset digits w_k = v_k + (p_k - 1)/2 >= 0
//      in 96-bit carry chains and normalises the chunk, keeping its carry.
// G3c: one block per 128 coefficients ripples the chunk carries, subtracts
//      floor(P/2) = sum_k (p_k - 1)/2 P_k and writes the two's-complement
//      32-bit limbs through shared memory in coalesced runs; G3cp: the same
//      with the chunks of few, long coefficients in parallel.
// G3f: all of it in one kernel for few primes.
#include <algorithm>

#include "../../include/rs.h"
#include "rs_internal.cuh"

namespace {

#include "tcdigits.cuh"  // store_digits8

__device__ __forceinline__ int32_t signed_rep3(uint32_t v, uint32_t p) {
  return v > (p >> 1) ? (int32_t)v - (int32_t)p : (int32_t)v;
}

__device__ __forceinline__ uint32_t finish64_3(int64_t s, const ModP &m) {
  return redc((uint64_t)(s + ((int64_t)m.p << 22)), m.p, m.pinv);  // 0 <= . < 2^54 < p 2^32
}

#define G3T_BK 64  // digits per digit block
#define G3T_SB 4   // digits per sub-block
#define G3T_LC 32  // earlier digits per staged chunk

// Digits by tiles: a block owns JT (32, or 16 when there are few coefficients
// to spread over the SMs) consecutive coefficients of one pair and produces
// their digits 64 at a time.  For the digit block [k0, k0 + 64) the
// contribution of every earlier digit,
//   A[k][j] = sum_{l < k0} W[k][l] v_l(j),
// is the product of a 64 x k0 slice of W and a k0 x JT slice of digits: chunks
// of both are staged in shared memory, and each of the 128 threads of a group
// accumulates 8 rows x JT/16 columns in int64.  |W|, |v| <= (p - 1) / 2, so 8
// products and a 32-bit rest stay below 2 (p - 1)^2 + 2^32 < 2^63; after every
// 8 the high words move to sums of their own (adds, while a fold by
// 2^32 mod p would take the multiply pipe that bounds the loop).  LS groups
// share the chunks of a block.
//
// The digits of the block then follow from the triangle of W inside it, with
// the constants folded in: S_k = (r_k - A[k]) c_k R, congruent to v_k R,
// W'[k][l] = -c_k W[k][l] (a table of 64 x 64 blocks, laid out as it is used)
// and h_k = (p_k - 1) / 2 give
//   v_k + h_k = REDC(S_k + h_k R + sum_{k0 <= l < k} W'[k][l] v_l)  in [0, p_k),
// so a digit waits for one REDC and one subtraction (about 45 cycles).  The 16
// threads that hold rows 4 s .. 4 s + 3 take the four digits of sub-block s in
// registers, right-looking; after a barrier the threads of later rows add
// these digits to their own sums (4 products and a fold per sum, independent;
// W' is loaded before the barrier).  Four digits a step, because the additions
// to eight rows a thread took longer than eight digits' chain.
// The block's residues, triangle and constants are copied to shared memory
// while its chunks are multiplied.
//
// What bounds it: this chain with few primes (before, one warp took all 64
// digits left-looking, 2,000 dependent product steps a block), the products
// with many.  Measured, before and now: see the choice of the digit kernels in
// engine.cu.
__device__ __forceinline__ void copy_async4(void *dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void copy_async16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

template <int JT, int LS>
__global__ void __launch_bounds__(128 * LS, 4 / LS) g3t_kernel(G3Args a) {
  constexpr int CJ = JT / 16;  // columns per thread
  // W[k0 + r][l0 + c] at Ws[.][c][r]: rows of 68 words keep eight consecutive r
  // 16-byte aligned (two shared loads) and the staging stores free of conflicts
  __shared__ __align__(16) int32_t Ws[LS][G3T_LC][G3T_BK + 4];
  __shared__ int32_t Vs[LS][G3T_LC][JT];                                 // digit l0 + c of coefficient j0 + jj
  __shared__ __align__(16) int32_t Wt[G3T_BK / G3T_SB][G3T_BK][G3T_SB];  // W'[k0 + r][k0 + 4 s + i], 4 s + i < r
  __shared__ int32_t Vb[G3T_BK][JT];                                     // the block's residues, then its digits
  __shared__ ModP Ms[G3T_BK];
  __shared__ uint32_t Cs[G3T_BK];
  constexpr int R = 8 / LS;  // rows per thread in the triangle: 8 rg + R grp + i
  static_assert(LS <= 2 && (LS == 1 || G3T_BK * JT * 8 <= (int)sizeof(Ws)), "the groups' sums fit in Ws");
  const int2 task = a.tasks[blockIdx.x];
  const PairDesc pd = a.pairs[task.x];
  const int K = pd.K, N = pd.N, S = pd.NI, j0 = task.y, tid = threadIdx.x;
  const int grp = tid >> 7, ltid = tid & 127, warp = ltid >> 5, lane = ltid & 31;
  const int rg = ltid >> 4, cg = ltid & 15;  // rows 8 rg .. 8 rg + 7, columns CJ cg .. CJ cg + CJ - 1
  uint32_t *col = a.coef + pd.img_off;       // residue, then digit, of (k, j) at col[k S + j]
  auto group_sync = [&] { asm volatile("bar.sync %0, 128;" ::"r"(grp + 1) : "memory"); };
  const int kend = a.kend ? min(K, a.kend) : K;
  for (int k0 = a.kbeg; k0 < kend; k0 += G3T_BK) {
    const int bk = min(G3T_BK, K - k0);
    // Chunks of W (16 rows of one column per thread) and digits are loaded into
    // registers one chunk ahead, so their latency overlaps the products.
    constexpr int NW = 16, NV = G3T_LC * JT / 128;
    int32_t wreg[NW], vreg[NV];
    const int wk = k0 + 16 * warp;  // the triangle of W has fewer than 2^27 entries (K <= 16384)
    const int32_t *wrow = a.wtab + wk * (wk - 1) / 2 + lane;
    const uint32_t *vcol = col + (size_t)(ltid / JT) * S + j0 + ltid % JT;
    const bool vlive = j0 + ltid % JT < N;
    auto fetch = [&](int l0) {
#pragma unroll
      for (int q = 0; q < NW; ++q)  // row wk + q starts q wk + q (q - 1) / 2 after row wk
        wreg[q] = wk + q < K ? __ldg(wrow + (l0 + q * wk + q * (q - 1) / 2)) : 0;
#pragma unroll
      for (int q = 0; q < NV; ++q) vreg[q] = vlive ? (int32_t)vcol[(size_t)(l0 + q * (128 / JT)) * S] : 0;
    };
    const int nch = (k0 - a.kbeg) / G3T_LC;  // k0 and kbeg are multiples of 64: full chunks
    if (grp < nch) fetch(a.kbeg + grp * G3T_LC);
    const int32_t *tri = a.wtri + (size_t)(k0 / G3T_BK) * (G3T_BK * G3T_BK);
#pragma unroll
    for (int e = tid; e < G3T_BK * G3T_BK / 4; e += 128 * LS) {  // piece (s, r): not all zero, and used
      const int r = e & 63;
      if (r < bk && r > 4 * (e >> 6)) copy_async16(&Wt[e >> 6][r][0], tri + 4 * e);
    }
#pragma unroll
    for (int e = tid; e < G3T_BK * JT; e += 128 * LS)
      if (e / JT < bk && j0 + e % JT < N) copy_async4(&Vb[e / JT][e % JT], col + (size_t)(k0 + e / JT) * S + j0 + e % JT);
    if (tid < G3T_BK) {  // rows past the last prime repeat it; their sums are never used
      copy_async16(&Ms[tid], a.mods + (k0 + min(tid, bk - 1)));
      copy_async4(&Cs[tid], a.crt + (k0 + min(tid, bk - 1)));
    }
    int64_t acc[8][CJ], high[8][CJ];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int c = 0; c < CJ; ++c) acc[i][c] = high[i][c] = 0;
    for (int ch = grp; ch < nch; ch += LS) {
#pragma unroll
      for (int q = 0; q < NW; q += 4)
        *reinterpret_cast<int4 *>(&Ws[grp][lane][16 * warp + q]) =
            make_int4(wreg[q], wreg[q + 1], wreg[q + 2], wreg[q + 3]);
#pragma unroll
      for (int q = 0; q < NV; ++q) Vs[grp][(ltid + 128 * q) / JT][ltid % JT] = vreg[q];
      group_sync();
      if (ch + LS < nch) fetch(a.kbeg + (ch + LS) * G3T_LC);
      if (16 * warp < bk) {
#pragma unroll 1
        for (int c0 = 0; c0 < G3T_LC; c0 += 8) {
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const int4 lo = *reinterpret_cast<const int4 *>(&Ws[grp][c0 + c][8 * rg]);
            const int4 hi = *reinterpret_cast<const int4 *>(&Ws[grp][c0 + c][8 * rg + 4]);
            const int32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
            for (int cc = 0; cc < CJ; ++cc) {
              const int64_t v = Vs[grp][c0 + c][CJ * cg + cc];
#pragma unroll
              for (int i = 0; i < 8; ++i) acc[i][cc] += w[i] * v;
            }
          }
#pragma unroll
          for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int cc = 0; cc < CJ; ++cc) {
              high[i][cc] += (int32_t)(acc[i][cc] >> 32);
              acc[i][cc] = (uint32_t)acc[i][cc];
            }
        }
      }
      group_sync();
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    // acc + 2^32 high, |high| < 2^42, congruent to a word below 2^56
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t c32 = Ms[8 * rg + i].r1;
#pragma unroll
      for (int cc = 0; cc < CJ; ++cc) acc[i][cc] += rs_fold64(high[i][cc], c32) * (int64_t)c32;
    }
    int64_t sum[R][CJ];
    if constexpr (LS > 1) {  // each group keeps R of a thread's rows; the others' sums go through the staging buffer
      int64_t *part = reinterpret_cast<int64_t *>(&Ws[0][0][0]);
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int cc = 0; cc < CJ; ++cc) {
          part[((grp * R + i) * CJ + cc) * 128 + ltid] = grp ? acc[i][cc] : acc[R + i][cc];
          sum[i][cc] = grp ? acc[R + i][cc] : acc[i][cc];
        }
      __syncthreads();
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int cc = 0; cc < CJ; ++cc) sum[i][cc] += part[(((1 - grp) * R + i) * CJ + cc) * 128 + ltid];
    } else {
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int cc = 0; cc < CJ; ++cc) sum[i][cc] = acc[i][cc];
    }
    // S + h R: (r - A) c R (plain r: W is in Montgomery form, its REDC removes R;
    // c in Montgomery form brings R back) as a folded word, plus h R mod p
    const int row0 = 8 * rg + R * grp;
    uint32_t rp[R], rpi[R], rc[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int r = row0 + i;
      const ModP m = Ms[r];
      const uint32_t c = Cs[r], hR = to_mont(m.p >> 1, m);
      rp[i] = m.p;
      rpi[i] = m.pinv;
      rc[i] = m.r1;
#pragma unroll
      for (int cc = 0; cc < CJ; ++cc) {
        const uint32_t res = r < bk && j0 + CJ * cg + cc < N ? (uint32_t)Vb[r][CJ * cg + cc] : 0u;
        const uint32_t A = redc((uint64_t)(sum[i][cc] + ((int64_t)m.p << 27)), m.p, m.pinv);  // |sum| < 2^57
        sum[i][cc] = rs_fold64((int64_t)((uint64_t)msub(res, A, m.p) * c), m.r1) + hR;
      }
    }
    __syncthreads();  // the residues in Vb are read: the digits take their place
    const int nsb = (bk + 3) / 4;
    for (int s = 0; s < nsb; ++s) {
#pragma unroll
      for (int q = 0; q < R; q += 4) {
        if (row0 + q != 4 * s) continue;
        int32_t w[4][4];  // w[r][i], i < r: W' of the sub-block's triangle
#pragma unroll
        for (int r = 1; r < 4; ++r) {
          const int4 x = *reinterpret_cast<const int4 *>(&Wt[s][4 * s + r][0]);
          w[r][0] = x.x, w[r][1] = x.y, w[r][2] = x.z;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
#pragma unroll
          for (int cc = 0; cc < CJ; ++cc) {
            // |sum| < 2^57 + 3 (p/2)^2: p 2^32 more if negative leaves [0, p 2^32)
            const uint32_t p = rp[q + i], h = (uint32_t)((uint64_t)sum[q + i][cc] >> 32);
            const uint32_t z = redc(((uint64_t)rs_umin(h, h + p) << 32) | (uint32_t)sum[q + i][cc], p, rpi[q + i]);
            const int32_t vs = (int32_t)z - (int32_t)(p >> 1);
#pragma unroll
            for (int r = i + 1; r < 4; ++r) sum[q + r][cc] += (int64_t)w[r][i] * vs;
            Vb[4 * s + i][CJ * cg + cc] = vs;
          }
        }
      }
      int4 w4[R];
#pragma unroll
      for (int i = 0; i < R; ++i) w4[i] = *reinterpret_cast<const int4 *>(&Wt[s][row0 + i][0]);
      __syncthreads();
      if (row0 + R > 4 * s + 4) {  // the later rows' sums, 4 products below (p/2)^2 each, folded
        int32_t v[4][CJ];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int cc = 0; cc < CJ; ++cc) v[i][cc] = Vb[4 * s + i][CJ * cg + cc];
#pragma unroll
        for (int i = 0; i < R; ++i) {
          if (R > 4 && row0 + i < 4 * s + 4) continue;
#pragma unroll
          for (int cc = 0; cc < CJ; ++cc) {
            int64_t t = (int64_t)w4[i].x * v[0][cc];
            t += (int64_t)w4[i].y * v[1][cc];
            t += (int64_t)w4[i].z * v[2][cc];
            t += (int64_t)w4[i].w * v[3][cc];
            sum[i][cc] += rs_fold64(t, rc[i]);
          }
        }
      }
    }
    // the digits over the residues (the last sub-block's barrier is behind)
#pragma unroll
    for (int e = tid; e < G3T_BK * JT; e += 128 * LS) {
      const int r = e / JT, j = j0 + e % JT;
      if (r < bk && j < N) col[(size_t)(k0 + r) * S + j] = (uint32_t)Vb[r][e % JT];
    }
    if (a.xdig) {  // and as operand digits of the tensor-core limb kernel
      uint16_t *x = a.xdig + pd.xd_off + (int64_t)(j0 >> 7) * ((K + 63) / 64) * 32768;
      for (int e = tid; e < G3T_BK / 8 * JT; e += 128 * LS) {
        const int r = 8 * (e / JT), jj = e % JT;
        if (r >= bk || j0 + jj >= N) continue;
        int32_t v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = r + i < bk ? Vb[r + i][jj] : 0;
        store_digits8(x, (j0 & 127) + jj, k0 + r, v);
      }
    }
    __syncthreads();  // this block's digits are read by the next digit blocks
  }
}

#define G3P_G 4     // digit rows per group
#define G3P_LC 128  // earlier digits per staged chunk of W

// Digits, one thread per coefficient: a block of 128 threads owns 128
// consecutive coefficients of one pair (the same tasks as the output
// kernel) and walks the digits in groups of 4 rows.  For the group
// [k0, k0 + 4) each thread accumulates A[k0 + i] = sum_{l < k0} W[k0 + i][l] v_l
// over its own earlier digits (re-read from the residue array they
// overwrote, where they stay in L1) with the four W values of each l
// broadcast from shared memory (one 16-byte load per l), lazily in int64 (a
// fold every 7 products); then it finishes the group's four digits in turn
// from the 4 x 4 triangle of W.  No warp waits for another: this is the form
// for batches with many coefficients, where one thread per coefficient
// fills the GPU (the tiled kernel serves batches with few coefficients and
// many primes).
__global__ void __launch_bounds__(128) g3p_kernel(G3Args a) {
  __shared__ __align__(16) int32_t Ws[G3P_LC][G3P_G];  // W[k0 + i][l0 + c] at Ws[c][i]
  __shared__ int32_t Wt[G3P_G][G3P_G];                 // W[k0 + i][k0 + c], c < i
  __shared__ ModP Ms[G3P_G];
  __shared__ uint32_t Cs[G3P_G];
  const int2 task = a.tasks[blockIdx.x];
  const PairDesc pd = a.pairs[task.x];
  const int K = pd.K, N = pd.N, S = pd.NI, t = (int)threadIdx.x, j = task.y + t;
  const bool live = j < N;
  uint32_t *col = a.coef + pd.img_off + (live ? j : 0);  // residue, then digit, of row k at col[k S]
  for (int k0 = 0; k0 < K; k0 += G3P_G) {
    const int g = min(G3P_G, K - k0);
    __syncthreads();  // the previous group's constants and triangle are no longer read
    if (t < G3P_G) {
      Ms[t] = a.mods[k0 + min(t, g - 1)];
      Cs[t] = a.crt[k0 + min(t, g - 1)];
    }
    if (t < G3P_G * G3P_G) {
      const int i = t >> 2, c = t & 3, k = k0 + i;
      Wt[i][c] = (c < i && i < g) ? __ldg(a.wtab + (size_t)k * (k - 1) / 2 + k0 + c) : 0;
    }
    int64_t acc[G3P_G] = {0, 0, 0, 0};
    uint32_t c32[G3P_G];
    for (int l0 = 0; l0 < k0; l0 += G3P_LC) {
      const int lc = min(G3P_LC, k0 - l0);
      if (l0 > 0) __syncthreads();  // the previous chunk is no longer read
#pragma unroll
      for (int i = 0; i < G3P_G; ++i) {  // row k0 + i, entries l0 + t
        const int k = k0 + i;
        Ws[t][i] = (t < lc && i < g) ? __ldg(a.wtab + (size_t)k * (k - 1) / 2 + l0 + t) : 0;
      }
      __syncthreads();
#pragma unroll
      for (int i = 0; i < G3P_G; ++i) c32[i] = Ms[i].r1;
      int c = 0;
      while (c < lc) {
        const int cend = min(c + 7, lc);  // 7 products per fold
#pragma unroll 7
        for (; c < cend; ++c) {
          const int32_t v = live ? (int32_t)col[(size_t)(l0 + c) * S] : 0;
          const int4 w = *reinterpret_cast<const int4 *>(&Ws[c][0]);
          acc[0] = rs_mac_s32(acc[0], w.x, v);
          acc[1] = rs_mac_s32(acc[1], w.y, v);
          acc[2] = rs_mac_s32(acc[2], w.z, v);
          acc[3] = rs_mac_s32(acc[3], w.w, v);
        }
#pragma unroll
        for (int i = 0; i < G3P_G; ++i) acc[i] = rs_fold64(acc[i], c32[i]);
      }
    }
    __syncthreads();  // Ms, Cs, Wt of this group are in place
    int32_t vg[G3P_G];
#pragma unroll
    for (int i = 0; i < G3P_G; ++i) {
      if (i >= g) break;
      const ModP m = Ms[i];
      int64_t s2 = rs_fold64(acc[i], m.r1);  // |s2| < 2^53
#pragma unroll
      for (int c = 0; c < i; ++c) s2 = rs_mac_s32(s2, Wt[i][c], vg[c]);  // + at most 3 products < 2^60
      s2 = rs_fold64(s2, m.r1);                                          // |s2| < 2^53 again
      const uint32_t r = live ? col[(size_t)(k0 + i) * S] : 0u;
      const uint32_t v = mmul(msub(r, finish64_3(s2, m), m.p), Cs[i], m);
      vg[i] = signed_rep3(v, m.p);
      if (live) col[(size_t)(k0 + i) * S] = (uint32_t)vg[i];
    }
  }
}

#ifndef RS_G3B_UNROLL
#define RS_G3B_UNROLL 4
#endif
constexpr int kG3bUnroll = RS_G3B_UNROLL;  // prime rows of the limb kernel per loop iteration

// Limb chunks: blockDim = 128 coefficients of one pair, one chunk of 16
// output limbs.  With the offset digits w_k = v_k + (p_k - 1)/2 in [0, p_k)
// the limb sums S[h] = sum_k w_k P_k[16 c + h] (P_k's 32-bit limbs) are
// unsigned and below K 2^63, so each is kept in a 96-bit carry chain; the
// chunk is then normalised into 16 limbs and a carry (< 2^47).  Only primes
// whose prefix product reaches this chunk contribute to it directly; lower
// terms arrive through the previous chunk's carry.
__global__ void __launch_bounds__(128) g3b_kernel(G3Args a) {
  const int4 task = a.ctasks[blockIdx.x];
  const PairDesc pd = a.pairs[task.x];
  const int c = task.z;
  const int j = task.y + (int)threadIdx.x;
  if (j >= pd.N) return;
  const int K = pd.K, N = pd.N;
  // first k whose prefix product has a limb in this chunk (nh is increasing)
  int lo = 0, hi = K;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (a.nh[mid] > 32 * c)
      hi = mid;
    else
      lo = mid + 1;
  }
  uint32_t a0[16], a1[16], a2[16];
#pragma unroll
  for (int h = 0; h < 16; ++h) a0[h] = a1[h] = a2[h] = 0u;
  const uint32_t *col = a.coef + pd.img_off + j;
#pragma unroll kG3bUnroll
  for (int k = lo; k < K; ++k) {
    const uint32_t half = (__ldg(&a.mods[k].p) - 1u) >> 1;
    const uint32_t w = (uint32_t)((int32_t)col[(size_t)k * pd.NI] + (int32_t)half);
    const uint4 *row = reinterpret_cast<const uint4 *>(a.p16 + __ldg(a.poff + k) + 32 * c);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint4 l4 = __ldg(row + q);
      rs_mac96(a0[4 * q], a1[4 * q], a2[4 * q], w, l4.x);
      rs_mac96(a0[4 * q + 1], a1[4 * q + 1], a2[4 * q + 1], w, l4.y);
      rs_mac96(a0[4 * q + 2], a1[4 * q + 2], a2[4 * q + 2], w, l4.z);
      rs_mac96(a0[4 * q + 3], a1[4 * q + 3], a2[4 * q + 3], w, l4.w);
    }
  }
  uint64_t carry = 0;
  uint32_t *xl = a.xl + pd.xl_off + j;
#pragma unroll
  for (int h = 0; h < 16; ++h) {
    const uint64_t lo64 = ((uint64_t)a1[h] << 32) | a0[h];
    const uint64_t t = lo64 + carry;
    const uint64_t ovf = t < lo64 ? 1u : 0u;
    xl[(size_t)(16 * c + h) * N] = (uint32_t)t;
    carry = (t >> 32) + (((uint64_t)a2[h] + ovf) << 32);
  }
  a.carry[pd.cy_off + (size_t)c * N + j] = (int64_t)carry;
}

// Carries and output: one thread per coefficient adds the chunk carries to
// the chunk limbs and subtracts floor(P / 2), P = p_0 ... p_{K-1} (the offset
// digits added sum_k (p_k - 1)/2 P_k = (P - 1)/2; limbs summed from the
// signed digits already have the symmetric value), giving the symmetric
// representative in two's complement; only the Lout low limbs are formed,
// which is exact because the result fits in them.  Each chunk's 16 limbs of
// the block's 128 coefficients are staged in shared memory and written back
// as runs of 16 consecutive limbs of one coefficient (out is
// [coefficient][limb], so a warp's store covers two 64-byte runs instead of
// 32 words Lout apart).  Also records the shape of each pair's result:
// shape[2 pair] = 1 + the largest index of a non-zero coefficient (0 for
// R = 0) and shape[2 pair + 1] = the most two's-complement limbs any
// coefficient needs (both by atomicMax on zeroed words).
__global__ void __launch_bounds__(128) g3c_kernel(G3Args a) {
  __shared__ uint32_t T[128 * 17];  // T[t * 17 + w]: limb 16 c + w of coefficient j0 + t
  const int2 task = a.tasks[blockIdx.x];
  const PairDesc pd = a.pairs[task.x];
  const int t = (int)threadIdx.x, j0 = task.y, j = j0 + t;
  const bool live = j < pd.N;
  const int N = pd.N, L = pd.Lout, C = (L + 15) / 16;
  const uint32_t *xl = a.xl + pd.xl_off + j;
  const int p0 = __ldg(a.poff + pd.K);
  const uint32_t *PK = reinterpret_cast<const uint32_t *>(a.p16 + p0);  // P's 32-bit limbs
  // limbs from the signed digits (tensor-core limb kernel) need no offset: P = 0 here
  const int plen = a.signed_digits ? 0 : (__ldg(a.poff + pd.K + 1) - p0) / 2;
  uint32_t *o = a.out + pd.out_off;
  int64_t r = 0;
  int last_nz = -1, last_nf = -1;  // last limb != 0, last limb != 0xffffffff
  uint32_t top_nz = 0u, top_nf = 0u, top = 0u;
  // A chunk's loads (its limbs, P's limbs, its carry) are independent of the
  // carry chain: chunk c + 1's are issued before chunk c's chain and stores,
  // so a chunk does not wait a memory latency after the previous one.
  auto load = [&](int c, uint32_t (&x)[16], uint32_t (&pkv)[17], int64_t &cyv) {
#pragma unroll
    for (int w = 0; w < 16; ++w) x[w] = xl[(size_t)(16 * c + w) * N];
#pragma unroll
    for (int w = 0; w < 17; ++w) pkv[w] = 16 * c + w < plen ? __ldg(PK + 16 * c + w) : 0u;
    cyv = a.carry[pd.cy_off + (size_t)c * N + j];
  };
  uint32_t xw[16], pk[17];
  int64_t cy = 0;
  if (live && C > 0) load(0, xw, pk, cy);
  for (int c = 0; c < C; ++c) {
    uint32_t xn[16], pn[17];
    int64_t cn = 0;
#pragma unroll
    for (int w = 0; w < 16; ++w) xn[w] = 0u;
#pragma unroll
    for (int w = 0; w < 17; ++w) pn[w] = 0u;
    if (live && c + 1 < C) load(c + 1, xn, pn, cn);
    if (live) {
#pragma unroll
      for (int w = 0; w < 16; ++w) {
        const int l = 16 * c + w;
        const uint32_t h = (pk[w] >> 1) | (pk[w + 1] << 31);
        const int64_t v = (int64_t)xw[w] + r - (int64_t)h;
        const uint32_t limb = (uint32_t)v;
        r = v >> 32;
        T[t * 17 + w] = limb;
        if (l < L) {
          if (limb != 0u) {
            last_nz = l;
            top_nz = limb;
          }
          if (limb != 0xffffffffu) {
            last_nf = l;
            top_nf = limb;
          }
          top = limb;
        }
      }
      r += cy;
    }
    __syncthreads();
    const int nl = min(16, L - 16 * c);  // limbs of this chunk that exist
#pragma unroll 4
    for (int q = 0; q < 16; ++q) {
      const int e = q * 128 + t, jj = e >> 4, w = e & 15;
      if (j0 + jj < N && w < nl) o[(size_t)(j0 + jj) * L + 16 * c + w] = T[jj * 17 + w];
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 16; ++w) xw[w] = xn[w];
#pragma unroll
    for (int w = 0; w < 17; ++w) pk[w] = pn[w];
    cy = cn;
  }
  if (!live) return;
  // fewest limbs whose two's-complement value is this coefficient
  const bool neg = (top >> 31) != 0u;
  if (!neg && last_nz < 0) return;  // a zero coefficient
  int need = neg ? last_nf + 1 + ((top_nf >> 31) ? 0 : 1) : last_nz + 1 + ((top_nz >> 31) ? 1 : 0);
  need = max(1, min(need, L));
  atomicMax(a.shape + 2 * task.x, j + 1);
  atomicMax(a.shape + 2 * task.x + 1, need);
}

// The same with the chunks of a coefficient in parallel, for few coefficients
// of many limbs:
// One thread per coefficient and chunk (lanes: 32 coefficients, so the loads
// are whole lines; threadIdx.y: blockDim.y chunks at a time; threadIdx.z:
// groups of 32 coefficients).  With the previous chunk's carry added, a chunk
// is W + 2^512 e0, 0 <= W < 2^512, and what it passes on is
//   f(e) = e0 + floor((W + e) / 2^512),  e in {-2, ..., 1} from the chunks below
// (the whole chunk is above -2^512 - 2^48 and below 2^512 + 2^48).  f's four
// values go to shared memory packed in a byte, every thread walks the bytes of
// the chunks below its own, adds its e, and the limbs leave through shared
// memory as runs of one coefficient (out is [coefficient][limb]).
//
// Bound by a few dependent latencies per step of blockDim.y chunks.  CRT stage,
// us, with one thread walking a coefficient's chunks -> here: 40 blocks of 122
// chunks 2,120 -> 2,036; 20 of 74 545 -> 489; 33 of 34 253 -> 225; 40 of 31
// 254 -> 229; 8 of 5 32.2 -> 30.3; but 4,899 blocks of 2 to 5 1,480 -> 1,630,
// 1,047 of one or two 34.4 -> 40.6, 512 of 33 1,790 -> 1,823 and one of one
// 16 -> 18 (short runs, more threads per limb): taken for three chunks or
// more and at most two blocks per SM.
constexpr int kG3cWords = 4 * 32 * (4 * 16 + 1);  // coefficients x (16 chunks' limbs + 1), over all splits

__global__ void __launch_bounds__(512) g3cp_kernel(G3Args a) {
  __shared__ uint32_t T[kG3cWords];  // T[t (16 G + 1) + 16 g + w]: limb 16 (c0 + g) + w of coefficient t
  __shared__ uint32_t fn[2][512];
  __shared__ int top[3][128];  // per coefficient: negative?, codes of the last limb != 0 and != 0xffffffff
  const int2 task = a.tasks[blockIdx.x];
  const PairDesc pd = a.pairs[task.x];
  const int G = (int)blockDim.y, lane = (int)threadIdx.x, g = (int)threadIdx.y;
  const int ct = (int)threadIdx.z * 32 + lane;  // coefficient of the block
  const int j0 = task.y + (int)(blockIdx.y * blockDim.z) * 32, j = j0 + ct;
  if (j0 >= pd.N) return;  // the whole block
  const bool live = j < pd.N;
  const int N = pd.N, L = pd.Lout, C = (L + 15) / 16, stride = 16 * G + 1;
  const uint32_t *xl = a.xl + pd.xl_off + j;
  const int64_t *cyp = a.carry + pd.cy_off + j;
  const int p0 = __ldg(a.poff + pd.K);
  const uint32_t *PK = reinterpret_cast<const uint32_t *>(a.p16 + p0);  // P's 32-bit limbs
  // limbs from the signed digits (tensor-core limb kernel) need no offset: P = 0 here
  const int plen = a.signed_digits ? 0 : (__ldg(a.poff + pd.K + 1) - p0) / 2;
  uint32_t *o = a.out + pd.out_off;
  if (g == 0) top[0][ct] = top[1][ct] = top[2][ct] = 0;
  __syncthreads();
  int e = 0;  // carry into the chunks of this step (equal for the threads of a coefficient)
  for (int c0 = 0; c0 < C; c0 += G) {
    const int c = c0 + g;
    const bool act = live && c < C;
    uint32_t x[16];
    uint32_t f = 0xe4u;  // the identity: f(e) = e
    if (act) {
      int64_t r = c ? cyp[(size_t)(c - 1) * N] : 0;
      uint32_t any = 0u, all = 0xffffffffu, rest = 0u, pk = 16 * c < plen ? __ldg(PK + 16 * c) : 0u;
#pragma unroll
      for (int w = 0; w < 16; ++w) x[w] = xl[(size_t)(16 * c + w) * N];
#pragma unroll
      for (int w = 0; w < 16; ++w) {
        const uint32_t pn = 16 * c + w + 1 < plen ? __ldg(PK + 16 * c + w + 1) : 0u;
        const uint32_t h = (pk >> 1) | (pn << 31);
        pk = pn;
        const int64_t v = (int64_t)x[w] + r - (int64_t)h;
        x[w] = (uint32_t)v;
        r = v >> 32;
        any |= x[w];
        all &= x[w];
        if (w) rest |= x[w];
      }
      const int e0 = (int)r + 2;
      f = (uint32_t)(e0 - (rest == 0u && x[0] < 2u ? 1 : 0)) | (uint32_t)(e0 - (any == 0u ? 1 : 0)) << 2 |
          (uint32_t)e0 << 4 | (uint32_t)(e0 + (all == 0xffffffffu ? 1 : 0)) << 6;
    }
    uint32_t *fs = fn[(c0 / G) & 1];
    fs[g * 32 * blockDim.z + ct] = f;
    __syncthreads();
    int mine = e;
    for (int i = 0; i < G; ++i) {
      if (i == g) mine = e;
      e = (int)((fs[i * 32 * blockDim.z + ct] >> (2 * (e + 2))) & 3u) - 2;
    }
    if (act) {
      int64_t r = mine;
      int nz = 0, nf = 0;  // 2 (index + 1) + whether the sign needs one more limb
#pragma unroll
      for (int w = 0; w < 16; ++w) {
        const int l = 16 * c + w;
        const int64_t v = (int64_t)x[w] + r;
        const uint32_t limb = (uint32_t)v;
        r = v >> 32;
        T[ct * stride + 16 * g + w] = limb;
        if (l < L) {
          if (limb != 0u) nz = 2 * (l + 1) + (int)(limb >> 31);
          if (limb != 0xffffffffu) nf = 2 * (l + 1) + (int)(~limb >> 31);
          if (l == L - 1) top[0][ct] = (int)(limb >> 31);
        }
      }
      atomicMax(&top[1][ct], nz);
      atomicMax(&top[2][ct], nf);
    }
    __syncthreads();
    const int nl = min(16 * G, L - 16 * c0);  // limbs of this step that exist
    for (int t = g; t < 32; t += G) {
      const int tt = (int)threadIdx.z * 32 + t;
      if (j0 + tt < N)
        for (int w = lane; w < nl; w += 32) o[(size_t)(j0 + tt) * L + 16 * c0 + w] = T[tt * stride + w];
    }
  }
  __syncthreads();
  if (g != 0) return;
  // fewest limbs whose two's-complement value is this coefficient
  const bool neg = top[0][ct] != 0;
  const int code = top[neg ? 2 : 1][ct];
  const bool zero = !live || (!neg && code == 0);
  const int need = zero ? 0 : max(1, min((code >> 1) + (code & 1), L));
  const int len = __reduce_max_sync(0xffffffffu, zero ? 0 : j + 1);
  const int most = __reduce_max_sync(0xffffffffu, need);
  if (lane == 0 && len) {
    atomicMax(a.shape + 2 * task.x, len);
    atomicMax(a.shape + 2 * task.x + 1, most);
  }
}

// The whole Chinese remaindering in one kernel for few primes (K <=
// RS_G3F_MAX_K): a thread owns a coefficient as in g3p_kernel, keeps its digits
// in a column of shared memory, forms each chunk of 16 limbs from them as in
// g3b_kernel and removes floor(P / 2) and writes the chunk out as in
// g3c_kernel, so neither digits nor limbs nor carries go through memory.
// Shared memory: digits [K][128]; W by groups of four rows, W[4 g + i][l] at
// 8 g (g - 1) + 4 l + i (l < 4 g: one 16-byte load gives four rows), then the
// groups' 4 x 4 triangles.
//
// Bound by launch latency and the chain of digits for few coefficients, by the
// products and the shared memory of a block for many.  Measured, against the
// three kernels: see the choice of the digit kernels in engine.cu.
__global__ void __launch_bounds__(128) g3f_kernel(G3Args a) {
  extern __shared__ __align__(16) int32_t fsm[];
  __shared__ ModP Ms[RS_G3F_MAX_K];
  __shared__ uint32_t Cs[RS_G3F_MAX_K];
  __shared__ uint32_t T[128 * 17];  // T[t * 17 + w]: limb 16 c + w of coefficient j0 + t
  const int2 task = a.tasks[blockIdx.x];
  const PairDesc pd = a.pairs[task.x];
  const int K = pd.K, N = pd.N, S = pd.NI, t = (int)threadIdx.x, j0 = task.y, j = j0 + t;
  const bool live = j < N;
  const int L = pd.Lout, C = (L + 15) / 16, ng = (K + 3) >> 2;
  int32_t *vs = fsm + t;                      // digit k at vs[128 k]
  int32_t *Wq = fsm + 128 * K, *Wt = Wq + 8 * ng * (ng - 1);
  const uint32_t *col = a.coef + pd.img_off + (live ? j : 0);
#pragma unroll 4
  for (int k = 0; k < K; ++k) vs[128 * k] = live ? (int32_t)col[(size_t)k * S] : 0;
  for (int k = t; k < K; k += 128) {
    Ms[k] = a.mods[k];
    Cs[k] = a.crt[k];
  }
  for (int k = t >> 5; k < 4 * ng; k += 4) {
    const int g = k >> 2, i = k & 3;
    const int32_t *row = a.wtab + k * (k - 1) / 2;
    for (int l = t & 31; l < 4 * g + 4; l += 32) {
      const int32_t w = l < k && k < K ? __ldg(row + l) : 0;
      if (l < 4 * g)
        Wq[8 * g * (g - 1) + 4 * l + i] = w;
      else
        Wt[16 * g + 4 * i + l - 4 * g] = w;
    }
  }
  __syncthreads();
  for (int g = 0; g < ng; ++g) {  // digits, four rows at a time
    const int k0 = 4 * g;
    int64_t acc[4] = {0, 0, 0, 0};
    const int4 *wq = reinterpret_cast<const int4 *>(Wq + 8 * g * (g - 1));
    uint32_t c32[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) c32[i] = Ms[min(k0 + i, K - 1)].r1;
    int l = 0;
    while (l < k0) {  // 4 products per fold: k0 is a multiple of 4
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int32_t v = vs[128 * (l + q)];
        const int4 w = wq[l + q];
        acc[0] = rs_mac_s32(acc[0], w.x, v);
        acc[1] = rs_mac_s32(acc[1], w.y, v);
        acc[2] = rs_mac_s32(acc[2], w.z, v);
        acc[3] = rs_mac_s32(acc[3], w.w, v);
      }
      l += 4;
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[i] = rs_fold64(acc[i], c32[i]);
    }
    int32_t vg[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (k0 + i >= K) break;
      const ModP m = Ms[k0 + i];
      int64_t s2 = acc[i];  // |s2| < 2^53
#pragma unroll
      for (int c = 0; c < i; ++c) s2 = rs_mac_s32(s2, Wt[16 * g + 4 * i + c], vg[c]);  // + at most 3 products < 2^60
      s2 = rs_fold64(s2, m.r1);
      const uint32_t v = mmul(msub((uint32_t)vs[128 * (k0 + i)], finish64_3(s2, m), m.p), Cs[k0 + i], m);
      vg[i] = signed_rep3(v, m.p);
      vs[128 * (k0 + i)] = vg[i];
    }
  }
  const int p0 = __ldg(a.poff + K);
  const uint32_t *PK = reinterpret_cast<const uint32_t *>(a.p16 + p0);  // P's 32-bit limbs
  const int plen = (__ldg(a.poff + K + 1) - p0) / 2;
  uint32_t *o = a.out + pd.out_off;
  int64_t r = 0;
  int lo = 0, nz = 0, nf = 0;  // nz, nf: 2 (1 + last limb != 0, != 0xffffffff) + whether the sign needs one more
  uint32_t top = 0u;
  for (int c = 0; c < C; ++c) {
    while (lo < K && __ldg(a.nh + lo) <= 32 * c) ++lo;  // prefix products below this chunk arrive as carries
    uint32_t a0[16], a1[16], a2[16];
#pragma unroll
    for (int h = 0; h < 16; ++h) a0[h] = a1[h] = a2[h] = 0u;
#pragma unroll 2
    for (int k = lo; k < K; ++k) {
      const uint32_t w = (uint32_t)(vs[128 * k] + (int32_t)((Ms[k].p - 1u) >> 1));
      const uint4 *row = reinterpret_cast<const uint4 *>(a.p16 + __ldg(a.poff + k) + 32 * c);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint4 l4 = __ldg(row + q);
        rs_mac96(a0[4 * q], a1[4 * q], a2[4 * q], w, l4.x);
        rs_mac96(a0[4 * q + 1], a1[4 * q + 1], a2[4 * q + 1], w, l4.y);
        rs_mac96(a0[4 * q + 2], a1[4 * q + 2], a2[4 * q + 2], w, l4.z);
        rs_mac96(a0[4 * q + 3], a1[4 * q + 3], a2[4 * q + 3], w, l4.w);
      }
    }
    uint64_t carry = 0;
    uint32_t pk = 16 * c < plen ? __ldg(PK + 16 * c) : 0u;
#pragma unroll
    for (int w = 0; w < 16; ++w) {
      const uint64_t lo64 = ((uint64_t)a1[w] << 32) | a0[w];
      const uint64_t x = lo64 + carry;
      carry = (x >> 32) + (((uint64_t)a2[w] + (x < lo64 ? 1u : 0u)) << 32);
      const uint32_t pn = 16 * c + w + 1 < plen ? __ldg(PK + 16 * c + w + 1) : 0u;
      const int64_t v = (int64_t)(uint32_t)x + r - (int64_t)((pk >> 1) | (pn << 31));
      pk = pn;
      const uint32_t limb = (uint32_t)v;
      r = v >> 32;
      T[t * 17 + w] = limb;
      const int l = 16 * c + w;
      if (l < L) {
        if (limb != 0u) nz = 2 * (l + 1) + (int)(limb >> 31);
        if (limb != 0xffffffffu) nf = 2 * (l + 1) + (int)(~limb >> 31);
        top = limb;
      }
    }
    r += (int64_t)carry;
    __syncthreads();
    const int nl = min(16, L - 16 * c);  // limbs of this chunk that exist
#pragma unroll 4
    for (int q = 0; q < 16; ++q) {
      const int e = q * 128 + t, jj = e >> 4, w = e & 15;
      if (j0 + jj < N && w < nl) o[(size_t)(j0 + jj) * L + 16 * c + w] = T[jj * 17 + w];
    }
    __syncthreads();
  }
  // fewest limbs whose two's-complement value is this coefficient
  const bool neg = (top >> 31) != 0u;
  const int code = neg ? nf : nz;
  const bool zero = !live || (!neg && code == 0);
  const int need = zero ? 0 : max(1, min((code >> 1) + (code & 1), L));
  const int len = __reduce_max_sync(0xffffffffu, zero ? 0 : j + 1);
  const int most = __reduce_max_sync(0xffffffffu, need);
  if ((t & 31) == 0 && len) {
    atomicMax(a.shape + 2 * task.x, len);
    atomicMax(a.shape + 2 * task.x + 1, most);
  }
}

// W[k][l] = p_0 ... p_{l-1} mod p_k (Montgomery form, signed), one thread per k.
__global__ void crt_w_kernel(const ModP *mods, int K, int32_t *wtab) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= K) return;
  const ModP m = mods[k];
  int32_t *w = wtab + (size_t)k * (k - 1) / 2;
  uint32_t acc = m.r1;
  for (int l = 0; l < k; ++l) {
    w[l] = signed_rep3(acc, m.p);
    acc = mmul(acc, to_mont(mods[l].p - m.p, m), m);  // p_l mod p_k (the table is descending)
  }
}

// The triangle of W inside each 64-prime block with -c_k folded in, as the
// tiled digit kernel copies it: -c_k W[k][l] (Montgomery form, signed) for
// k = 64 b + r, l = 64 b + 4 s + i < k at [b][s][r][i], zero elsewhere.
__global__ void crt_tri_kernel(const ModP *mods, const uint32_t *crt, const int32_t *wtab, int K, int32_t *wtri) {
  const int b = blockIdx.x;
  for (int e = threadIdx.x; e < G3T_BK * G3T_BK; e += blockDim.x) {
    const int s = e >> 8, r = (e >> 2) & 63, c = 4 * s + (e & 3), k = G3T_BK * b + r;
    int32_t w = 0;
    if (c < r && k < K) {
      const ModP m = mods[k];
      const int32_t x = wtab[(size_t)k * (k - 1) / 2 + G3T_BK * b + c];
      w = signed_rep3(mmul(x < 0 ? (uint32_t)(-x) : m.p - (uint32_t)x, crt[k], m), m.p);
    }
    wtri[(size_t)b * (G3T_BK * G3T_BK) + e] = w;
  }
}

// One warp per (factor, prime): g mod p by Horner over g's limbs
// (r <- r 2^32 + limb, with 2^32 = R mod p taken as mmul by R^2 mod p), its
// inverse by Fermat, then the factor's residues times that inverse (plain
// residues times a Montgomery-form value stay plain).  g = 0 mod p gives 0.
__global__ void scale_kernel(const ScaleDesc *sd, int nf, int kmax, const ModP *mods, const uint32_t *gw,
                             const uint32_t *in, uint32_t *out) {
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (warp >= (int64_t)nf * kmax) return;
  const int fi = (int)(warp / kmax), k = (int)(warp - (int64_t)fi * kmax);
  const ScaleDesc d = sd[fi];
  if (k >= d.k) return;
  const ModP m = mods[k];
  uint32_t r = 0u;
  for (int l = d.g_len - 1; l >= 0; --l) {
    uint32_t limb = gw[d.g_off + l];  // < 2^32 < 4p
    while (limb >= m.p) limb -= m.p;
    r = madd(mmul(r, m.r2, m), limb, m.p);
  }
  const uint32_t inv = minv(to_mont(r, m), m);
  const uint32_t *src = in + d.src_off + (int64_t)k * d.src_stride;
  uint32_t *dst = out + d.dst_off + (int64_t)k * d.n;
  for (int j = lane; j < d.n; j += 32) dst[j] = mmul(src[j], inv, m);
}

}  // namespace

cudaError_t launch_scale(const ScaleDesc *sd, int nf, int kmax, const ModP *mods, const uint32_t *gw,
                         const uint32_t *in, uint32_t *out, cudaStream_t s) {
  const int64_t warps = (int64_t)nf * kmax;
  if (warps > 0) scale_kernel<<<(unsigned)((warps + 3) / 4), 128, 0, s>>>(sd, nf, kmax, mods, gw, in, out);
  return cudaGetLastError();
}

cudaError_t launch_g3t(int nt, const G3Args &a, const int2 *ttasks, cudaStream_t s, int jt) {
  G3Args at = a;
  at.tasks = ttasks;
  if (nt) {
    if (jt == 16)
      g3t_kernel<16, 2><<<nt, 256, 0, s>>>(at);
    else
      g3t_kernel<32, 1><<<nt, 128, 0, s>>>(at);
  }
  return cudaGetLastError();
}

cudaError_t launch_g3p(int nt, const G3Args &a, const int2 *tasks, cudaStream_t s) {
  G3Args at = a;
  at.tasks = tasks;
  if (nt) g3p_kernel<<<nt, 128, 0, s>>>(at);
  return cudaGetLastError();
}

static size_t g3f_smem(int kmax) {
  const int ng = (kmax + 3) / 4;
  return (size_t)(128 * kmax + 8 * ng * (ng - 1) + 16 * ng) * 4;
}

cudaError_t g3f_prepare() {
  return cudaFuncSetAttribute(g3f_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g3f_smem(RS_G3F_MAX_K));
}

cudaError_t launch_g3f(int nc, int kmax, const G3Args &a, const int2 *otasks, cudaStream_t s) {
  G3Args ao = a;
  ao.tasks = otasks;
  const size_t smem = g3f_smem(kmax);
  if (nc) g3f_kernel<<<nc, 128, smem, s>>>(ao);
  return cudaGetLastError();
}

cudaError_t launch_g3bc(int nb, int nc, int maxL, int sms, const G3Args &a, const int2 *otasks, cudaStream_t s) {
  if (nb) g3b_kernel<<<nb, 128, 0, s>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  G3Args ao = a;
  ao.tasks = otasks;
  // Chunks in parallel: 16 (chunk, 32 coefficients) groups a block, as many
  // chunks at once as the longest coefficient has, the 128 coefficients of a
  // task in 1, 2 or 4 parts.
  const int C = (maxL + 15) / 16, G = std::max(1, std::min(16, C)), Z = G <= 4 ? 4 : G <= 8 ? 2 : 1;
  if (nc && C >= 3 && nc <= 2 * sms)
    g3cp_kernel<<<dim3(nc, 4 / Z), dim3(32, G, Z), 0, s>>>(ao);
  else if (nc)
    g3c_kernel<<<nc, 128, 0, s>>>(ao);
  return cudaGetLastError();
}

int64_t crt_tri_words(int K) { return (int64_t)((K + G3T_BK - 1) / G3T_BK) * (G3T_BK * G3T_BK); }

cudaError_t launch_crt_tables(const ModP *mods, const uint32_t *crt, int K, int32_t *wtab, int32_t *wtri,
                              cudaStream_t s) {
  crt_w_kernel<<<(K + 63) / 64, 64, 0, s>>>(mods, K, wtab);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  crt_tri_kernel<<<(K + G3T_BK - 1) / G3T_BK, 256, 0, s>>>(mods, crt, wtab, K, wtri);
  return cudaGetLastError();
}
