// G1: fused modular reduction + evaluation + univariate resultant, one
// thread per modular image (pair, prime p, point x_i).  Paper, Section 4.1:
// Collins' algorithm maps f, g to Z_p and evaluates them at points x_i
// (steps 1-2), then takes z_i^{(p)} = res(f(x_i, y), g(x_i, y), y) in Z_p.
// The points come in pairs +-q^i (q of multiplicative order above the
// largest point count, chosen per prime).  With f_j(x) = E_j(x^2) + x O_j(x^2)
// (even and odd parts), both images of a pair need E_j(Q^i) and x O_j(Q^i)
// only, Q = q^2, x = q^i: the sums of f_{j,k} q^{ik} over the even and over
// the odd k.  The two threads of a pair each take one parity, as a
// correlation of chirp-scaled coefficients with the sequence q^{C(t,2)}
// (accumulated without per-term reduction), and exchange it with a shuffle:
// f_j(+-q^i) = E_j(Q^i) +- q^i O_j(Q^i).  G2 splits the images back into
// E and O and interpolates each with two convolutions.
//
// The univariate resultant keeps the formal degrees (a, b) = (m_y, n_y) of
// the Sylvester matrix of Section 3.1, so z_i^{(p)} = R^{(y)}(x_i) mod p for
// every prime and point.  It is computed by a division-free remainder
// sequence on the two coefficient vectors held in registers, top-aligned
// (index 0 = leading coefficient), with one final inversion left to G2:
//
//   a >= b, l_B != 0:  A' = l_B A - l_A y^(a-b) B  (top term cancels, formal
//                      degree a-1);  Res_{a,b}(A,B) l_B^{b-1} = (-1)^b Res_{a-1,b}(A',B)
//   a <  b, l_A != 0:  B' = l_A B - l_B y^(b-a) A;  Res_{a,b}(A,B) l_A^{a-1} = Res_{a,b-1}(A,B')
//   a >= b, l_B == 0:  Res_{a,b}(A,B) = l_A Res_{a,b-1}(A, B without its zero top)
//   a <  b, l_A == 0:  Res_{a,b}(A,B) = (-1)^b l_B Res_{a-1,b}(A without its zero top, B)
//   Res_{0,b}(A,B) = A_0^b,  Res_{a,0}(A,B) = B_0^a
//
// (each identity is a row operation on the Sylvester matrix followed by a
// cofactor expansion along its first column).  Two steps in a row reduce the
// same polynomial whenever a >= b + 1 (pivot l_B twice), and they are taken in
// one pass over its coefficients:
//
//   a >= b + 1, l_B != 0:  A'' = l_B^2 A - (alpha y + beta) y^(a-b-1) B,
//     alpha = l_B A_0, beta = l_B A_1 - A_0 B_1 (index = power below the top);
//     Res_{a,b}(A,B) (l_B^2)^{b-1} = Res_{a-2,b}(A'',B), and the same on B.
//
// In the normal sequence (degrees one apart) every pass is of this kind: three
// products and one Montgomery reduction per coefficient for two degrees,
// against four products and two reductions in single steps.  The three
// multipliers c (each below p) are negated together when their sum exceeds
// 2^32, so that their products with residues stay below 2^32 p and one
// unsigned REDC finishes the sum; a pass on A negated so gives
// (-1)^b Res(A'', B).
//
// The pivot powers prod_t c_t^{e_t} (c the pivot of a single step, e its
// degree minus one; the square of the pivot in a double step) have
// non-increasing e_t, so they are accumulated by Abel summation: with
// Q_t = c_1 ... c_t, prod_t c_t^{e_t} = prod_t Q_t^{e_t - e_{t+1}}: one product
// per pass into Q and one into the denominator whenever e drops.
//
// Register arrays have a compile-time capacity C; once both degrees fit in
// C - S entries (S = RS_G1_PSTEP) the state moves to arrays of C - S (registers
// are renamed, nothing is copied), so the unrolled update loops shrink with
// the degrees.
//
// Bound: the multiply pipe.  A wide product costs 4.2 issue cycles per warp
// and SM partition, a low one 2.1: 19.5 cycles per coefficient of a double
// pass against 2 x 15.2 in single steps (both measured with 16 warps per SM
// on arrays of 24).  G1 on batches of 16 pairs with deg_x = 24, 32-bit
// coefficients, ns per image with single and with double steps:
//   deg_y       14     22     28     38     44     52     60     68
//   single   0.305  0.460  0.653  0.998  1.302  1.756  2.297  2.550
//   double   0.284  0.404  0.578  0.817  1.075  1.389  1.802  2.081
// (the evaluation is in both).
#include "rs_internal.cuh"

// Register capacity dropped per phase (S), entries per length check of a
// double step (T) and minimum resident 128-thread blocks per SM requested from
// ptxas (caps registers at 65536 / (128 * MINB) per thread), per capacity C.
// A phase costs code (two unrolled double steps; with many phases the warps
// miss the instruction cache: at C = 56 "no instruction" took 19% of the
// stalls with S = 12, 7% with 28), a longer phase more length checks.
// ns per image, deg_y = C - 4 (C - 2 at 16, 24 and 40):
//   C                    16     24     32     40     48     56     64     72
//   S = 12, T = 2     0.289  0.426  0.573  0.886  1.152  1.503  2.006  2.098
//   S = 16, T = 2     0.282  0.438  0.562  0.849  1.099  1.459  1.899  2.113
//   S = 20, T = 4     0.288  0.415  0.569  0.815  1.097  1.412  1.844  2.103
//   S = 28, T = 4     0.292  0.416  0.573  0.846  1.075  1.386  1.795  2.110
//   5 blocks, S = 12  0.291  0.402  0.571  0.909  1.251
#ifndef RS_G1_PSTEP
#define RS_G1_PSTEP (RS_G1_CAP <= 8 ? 8 : RS_G1_CAP <= 16 ? 16 : RS_G1_CAP <= 24 ? 12 : RS_G1_CAP <= 32 ? 16 \
                     : RS_G1_CAP <= 40 ? 20 : RS_G1_CAP <= 64 ? 28 : 12)
#endif
#ifndef RS_G1_TAIL
#define RS_G1_TAIL (RS_G1_CAP <= 32 || RS_G1_CAP > 64 ? 2 : 4)
#endif
#ifndef RS_G1_MINB
#define RS_G1_MINB (RS_G1_CAP <= 16 ? 6 : RS_G1_CAP <= 24 ? 5 : RS_G1_CAP <= 48 ? 4 : 3)
#endif

namespace {

struct Prs {
  int a, b;        // formal degrees of A and B
  uint32_t num;    // numerator (Montgomery form)
  uint32_t den;    // accumulated pivot powers (Montgomery form)
  uint32_t Q;      // running product of pivots
  int eprev;       // exponent of the previous pivot
  uint32_t sign;   // parity of the accumulated (-1) factors
  uint32_t degen;  // a zero pivot was met
};

__device__ __forceinline__ void settle(Prs &s, int e, uint32_t c, const ModP &m) {
  while (s.eprev > e) {
    s.den = mmul(s.den, s.Q, m);
    --s.eprev;
  }
  s.Q = mmul(s.Q, c, m);
  s.eprev = e;
}

// Entries I .. C - 2 of a reduction whose result has `live` entries: entry
// I is computed while I < live, entry `live` (the old constant term shifted
// out) becomes zero, and the zero padding beyond it is left alone.  The
// degrees are the same for every image of a tile, so these branches are
// uniform across the warp and skip the padding instead of multiplying zeros.
template <int C, int I>
__device__ __forceinline__ void reduce_tail(uint32_t (&P)[C], const uint32_t (&V)[C], uint32_t w1, uint32_t w2,
                                            const ModP &m, int live) {
  if constexpr (I < C - 1) {
    if (live > I) {
      P[I] = mmul2(P[I + 1], w1, V[I + 1], w2, m);
      reduce_tail<C, I + 1>(P, V, w1, w2, m, live);
    } else {
      P[I] = 0u;
    }
  }
}

// P[i] <- w1 P[i+1] + w2 V[i+1] for i < live (the reduced polynomial's
// entries); the top entry (which cancels) is dropped.  Every caller reduces
// an array whose degree is at least C - S (the phase condition), so the
// first C - S entries are always live and only the last S - 1 are checked.
template <int C>
__device__ __forceinline__ void reduce_into(uint32_t (&P)[C], const uint32_t (&V)[C], uint32_t w1,
                                            uint32_t w2, const ModP &m, int live) {
  constexpr int H = C > RS_G1_PSTEP ? C - RS_G1_PSTEP : 0;
#pragma unroll
  for (int i = 0; i < H; ++i) P[i] = mmul2(P[i + 1], w1, V[i + 1], w2, m);
  reduce_tail<C, H>(P, V, w1, w2, m, live);
  P[C - 1] = 0u;
}

// Entry I of a double step.
template <int C, int I>
__device__ __forceinline__ void reduce2_entry(uint32_t (&P)[C], const uint32_t (&V)[C], uint32_t c2, uint32_t c1,
                                              uint32_t c0, const ModP &m) {
  if constexpr (I < C - 2)
    P[I] = redc((uint64_t)P[I + 2] * c2 + (uint64_t)V[I + 2] * c1 + (uint64_t)V[I + 1] * c0, m.p, m.pinv);
  else if constexpr (I < C)
    P[I] = 0u;
}

template <int C, int I, int E>
__device__ __forceinline__ void reduce2_entries(uint32_t (&P)[C], const uint32_t (&V)[C], uint32_t c2, uint32_t c1,
                                                uint32_t c0, const ModP &m) {
  if constexpr (I < E) {
    reduce2_entry<C, I>(P, V, c2, c1, c0, m);
    reduce2_entries<C, I + 1, E>(P, V, c2, c1, c0, m);
  }
}

// Entries I .. C - 1 of a double step whose result has `live` entries, in
// groups; a group that is not computed holds only the two entries shifted
// out, which become zero (computed entries past the length come out zero).
template <int C, int I>
__device__ __forceinline__ void reduce2_tail(uint32_t (&P)[C], const uint32_t (&V)[C], uint32_t c2, uint32_t c1,
                                             uint32_t c0, const ModP &m, int live) {
  if constexpr (I < C) {
    if (live > I) {
      reduce2_entries<C, I, I + RS_G1_TAIL>(P, V, c2, c1, c0, m);
      reduce2_tail<C, I + RS_G1_TAIL>(P, V, c2, c1, c0, m, live);
    } else {
      P[I] = 0u;
      if constexpr (I + 1 < C) P[I + 1] = 0u;
    }
  }
}

// P[i] <- c2 P[i+2] + c1 V[i+2] + c0 V[i+1] for i < live: two steps on P, the
// two top entries (which cancel) dropped.  c2 + c1 + c0 <= 2^32.  Callers
// reduce a degree of at least C - S (S the phase), so live >= C - S - 1.
template <int C>
__device__ __forceinline__ void reduce2_into(uint32_t (&P)[C], const uint32_t (&V)[C], uint32_t c2, uint32_t c1,
                                             uint32_t c0, const ModP &m, int live) {
  constexpr int H = C > RS_G1_PSTEP ? C - RS_G1_PSTEP - 1 : 0;
  reduce2_entries<C, 0, H>(P, V, c2, c1, c0, m);
  reduce2_tail<C, H>(P, V, c2, c1, c0, m, live);
}

template <int C>
__device__ __forceinline__ void drop_top(uint32_t (&P)[C]) {
#pragma unroll
  for (int i = 0; i < C - 1; ++i) P[i] = P[i + 1];
  P[C - 1] = 0u;
}

// One normal step on A (a >= b, l_B != 0).
template <int C>
__device__ __forceinline__ void step_a(uint32_t (&A)[C], const uint32_t (&B)[C], Prs &s, const ModP &m) {
  const uint32_t lb = B[0], la = A[0];
  settle(s, s.b - 1, lb, m);
  reduce_into<C>(A, B, lb, mneg(la, m.p), m, s.a);
  s.sign ^= (uint32_t)(s.b & 1);
  --s.a;
}

// Two steps at once on P (formal degree d, reduced) with V (formal degree
// e <= d - 1, pivot V[0] != 0): returns 1 if the result was negated.
template <int C>
__device__ __forceinline__ uint32_t step2(uint32_t (&P)[C], const uint32_t (&V)[C], int d, int e, Prs &s,
                                          const ModP &m) {
  const uint32_t lv = V[0], np0 = m.p - P[0];  // in (0, p]
  uint32_t c2 = mmul(lv, lv, m);
  settle(s, e - 1, c2, m);
  uint32_t c1 = mmul(lv, np0, m);                         // -lv P_0
  uint32_t c0 = mmul2(P[0], V[1], m.p - lv, P[1], m);     // P_0 V_1 - lv P_1
  // halves: a sum below 2^31 - 1 bounds c2 + c1 + c0 by 2^32 - 1; otherwise
  // the negated sum is at most 3 p - (2^32 - 2) < 2^31 + 2
  const uint32_t neg = (c2 >> 1) + (c1 >> 1) + (c0 >> 1) >= 0x7fffffffu ? 1u : 0u;
  if (neg) {
    c2 = m.p - c2;
    c1 = m.p - c1;
    c0 = m.p - c0;
  }
  reduce2_into<C>(P, V, c2, c1, c0, m, d - 1);
  return neg;
}

template <int C>
__device__ __forceinline__ void prs_run(uint32_t (&A)[C], uint32_t (&B)[C], Prs &s, const ModP &m) {
  // invariant: a, b <= C - 1
  constexpr int S = RS_G1_PSTEP;
  // Fast path: double steps on the polynomial of larger degree (after one
  // single step if the degrees are equal), until a pivot vanishes or both
  // degrees fit the next phase.
  for (;;) {
    if (s.a == s.b) {
      if (s.a < 1 || B[0] == 0u || (C > S && s.a <= C - S - 1)) break;
      step_a<C>(A, B, s, m);
    }
    if (s.b > s.a) {
      if (s.a < 1 || A[0] == 0u || (C > S && s.b <= C - S - 1)) break;
      const uint32_t neg = step2<C>(B, A, s.b, s.a, s, m);
      s.sign ^= neg & (uint32_t)s.a;
      s.b -= 2;
    }
    if (s.a > s.b) {
      if (s.b < 1 || B[0] == 0u || (C > S && s.a <= C - S - 1)) break;
      const uint32_t neg = step2<C>(A, B, s.a, s.b, s, m);
      s.sign ^= neg & (uint32_t)s.b;
      s.a -= 2;
    }
  }
  // General steps: zero pivots, the last steps, and the phase boundary.
  while (s.a > 0 && s.b > 0 && (C <= S || s.a > C - S - 1 || s.b > C - S - 1)) {
    if (s.a >= s.b) {
      const uint32_t lb = B[0];
      if (lb != 0u) {
        const uint32_t la = A[0];
        settle(s, s.b - 1, lb, m);
        reduce_into<C>(A, B, lb, mneg(la, m.p), m, s.a);
        s.sign ^= (uint32_t)(s.b & 1);
        --s.a;
      } else {
        s.num = mmul(s.num, A[0], m);
        drop_top<C>(B);
        --s.b;
        s.degen = 1u;
      }
    } else {
      const uint32_t la = A[0];
      if (la != 0u) {
        const uint32_t lb = B[0];
        settle(s, s.a - 1, la, m);
        reduce_into<C>(B, A, la, mneg(lb, m.p), m, s.b);
        --s.b;
      } else {
        s.num = mmul(s.num, B[0], m);
        s.sign ^= (uint32_t)(s.b & 1);
        drop_top<C>(A);
        --s.a;
        s.degen = 1u;
      }
    }
  }
  if constexpr (C > S) {
    if (s.a > 0 && s.b > 0) {
      uint32_t A2[C - S], B2[C - S];
#pragma unroll
      for (int i = 0; i < C - S; ++i) {
        A2[i] = A[i];
        B2[i] = B[i];
      }
      prs_run<C - S>(A2, B2, s, m);
      return;
    }
  }
  if (s.a == 0)
    s.num = mmul(s.num, mpow(A[0], (uint32_t)s.b, m), m);
  else
    s.num = mmul(s.num, mpow(B[0], (uint32_t)s.a, m), m);
}

// Montgomery form of a two's-complement limb integer:
// sum_l limb_l 2^(32 l) R - [negative] 2^(32 L) R, with V[l] = 2^(32 l) R^2.
__device__ __forceinline__ uint32_t reduce_coef(const uint32_t *src, int L, const uint32_t *V,
                                                const ModP &m) {
  uint32_t acc = 0u;
  for (int l = 0; l < L; ++l) acc = madd(acc, redc((uint64_t)src[l] * V[l], m.p, m.pinv), m.p);
  if (src[L - 1] >> 31) acc = msub(acc, redc((uint64_t)V[L], m.p, m.pinv), m.p);
  return acc;
}

// The same for many limbs (L <= 128): the products are summed exactly in 96
// bits, one multiply a limb, and reduced once.
__device__ __forceinline__ uint32_t reduce_long(const uint32_t *src, int L, const uint32_t *V, const ModP &m) {
  uint32_t a0 = 0u, a1 = 0u, a2 = 0u;
  for (int l = 0; l < L; ++l) rs_mac96(a0, a1, a2, src[l], V[l]);
  uint64_t t = (uint64_t)a2 * m.r1 + a1;  // a2 < 2^7, 2^32 mod p <= 2^21: t < 2^32 + 2^28 < 3 p
  if (t >= 2ull * m.p) t -= 2ull * m.p;
  const uint32_t h = rs_umin((uint32_t)t, (uint32_t)t - m.p);
  uint32_t acc = redc(((uint64_t)h << 32) | a0, m.p, m.pinv);
  if (src[L - 1] >> 31) acc = msub(acc, redc((uint64_t)V[L], m.p, m.pinv), m.p);
  return acc;
}

__device__ __forceinline__ int32_t signed_rep(uint32_t v, uint32_t p) {
  return v > (p >> 1) ? (int32_t)v - (int32_t)p : (int32_t)v;
}

// Evaluation of the sum over the k of parity par (0 even, 1 odd) at x = q^i
// by the chirp identity i k = C(i+k,2) - C(i,2) - C(k,2):
//   sum_{k = par mod 2} f_{j,k} q^{ik} = q^{-C(i,2)} sum_{k = par mod 2} (f_{j,k} q^{-C(k,2)}) q^{C(i+k,2)},
// which is E_j(Q^i) for par = 0 and x O_j(Q^i) for par = 1.  The factor
// w_i = q^{-C(i,2)} is the same for every coefficient of f and g at the point
// pair, and the Sylvester determinant is homogeneous of degree n_y in the
// f-entries and m_y in the g-entries, so the coefficients are left without
// it and the image is multiplied by w_i^(m_y + n_y) at the end.  The staged
// coefficients a[k][r] = f_{deg-r,k} q^{-C(k,2)} (top-aligned in r, zero past
// the degree) and the window w[t] = q^{C(x0+t,2)} are signed representatives
// (|v| < 2^30), so 7 products stay below 7 2^60 in magnitude.  The sums are
// unsigned 64-bit words that start at p 2^32 (0 mod p, and above 7 2^60), so
// they never go below zero; after every 7 rows a fold hi 2^32 + lo ->
// hi (2^32 mod p) + lo + p 2^32 (2^32 mod p <= 2^21 for every table prime)
// starts the next.  At the end the high word, below 2 p, loses p if it can,
// which leaves less than p 2^32 for one REDC.
//
// One rolled loop over blocks of 8 columns serves every block of f and g: the
// values go through the thread's own shared-memory column, which is read back
// into the register array.  Fully unrolled over the register array the
// evaluation was more code than the remainder sequence, most of it not
// products: limits read per column, sums cleared and finished, signs and
// selects around the shuffle (6,026 instructions per warp and chunk at
// deg_x 24, deg_y 36, now under 4,500, of which 1,000 are products).
// G1 with deg_x = 24, ns per image, unrolled and now (double steps in both):
//   deg_y       14     22     28     38     44     52     60     68
//   unrolled 0.284  0.404  0.578  0.817  1.075  1.389  1.802  2.081
//   rolled   0.265  0.363  0.512  0.742  0.978  1.237  1.593  1.845
// Signed sums that start at 0 (8 rows before the first fold) measured 1-3%
// slower beyond 8 rows and 2% faster up to them.
//
// The columns are (C + 1) words a thread.  Inputs whose staged coefficients
// leave too little room beside them (the rule and both sides' times: engine.cu,
// rs_g1_column) take the form without (COL false): the same loop, each block's
// values selected into the register array; at most two blocks fit an SM then,
// so a thread may have 255 registers.

// Rows of one parity of a polynomial of x-degree mx (both parities have the
// same number; the last row may be a zero row), and the distance in words
// between the two parities: 16 mod 32, so that the two lanes of a point pair
// read different banks.
__host__ __device__ __forceinline__ int g1_half_rows(int mx) { return (mx >> 1) + 1; }
__host__ __device__ __forceinline__ int g1_odd_offset(int mx, int C) {
  const int w = g1_half_rows(mx) * C;
  return w + ((48 - (w & 31)) & 31);
}
__host__ __device__ __forceinline__ int g1_poly_words(int mx, int C) { return g1_odd_offset(mx, C) + g1_half_rows(mx) * C; }

// Values of f_j (or g_j) at +q^i (lane par = 0) and, negated, at -q^i (lane
// par = 1), j from the top: E + xO and xO - E from the partner lane's part.
// The sign of the second is the same for every coefficient of f and g; the
// image takes it back.  sa: staged coefficients of this lane's parity; steps:
// rows per block of 8 columns; win: the window at this point pair and parity;
// col: this thread's C words of shared memory (COL).
template <int C, bool COL>
__device__ __forceinline__ void eval_chirp(uint32_t (&P)[C], const int32_t *sa, const int32_t *steps,
                                           const int32_t *win, uint32_t *col, int par, const ModP &m) {
  const uint32_t c32 = m.r1;  // 2^32 mod p
  const uint32_t sg = par ? 1u : 0u - 1u, off = par ? 0u : m.p;  // sent: O, or p - E
  uint32_t *pc = col;
#pragma unroll 1
  for (int b = 0; b < C / 8; ++b) {
    const int32_t *pa = sa + 8 * b;
    const int32_t *pw = win;
    uint64_t acc[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) acc[r] = (uint64_t)m.p << 32;
    auto step = [&](int u) {
      const int64_t c = pw[2 * u];
      const int4 lo = *reinterpret_cast<const int4 *>(pa + u * C);
      const int4 hi = *reinterpret_cast<const int4 *>(pa + u * C + 4);
      acc[0] += (uint64_t)(lo.x * c);
      acc[1] += (uint64_t)(lo.y * c);
      acc[2] += (uint64_t)(lo.z * c);
      acc[3] += (uint64_t)(lo.w * c);
      acc[4] += (uint64_t)(hi.x * c);
      acc[5] += (uint64_t)(hi.y * c);
      acc[6] += (uint64_t)(hi.z * c);
      acc[7] += (uint64_t)(hi.w * c);
    };
    int n = steps[b];
#pragma unroll 1
    for (; n >= 7; n -= 7) {
#pragma unroll
      for (int u = 0; u < 7; ++u) step(u);
      pa += 7 * C;
      pw += 14;
#pragma unroll
      for (int r = 0; r < 8; ++r)
        acc[r] = (acc[r] >> 32) * c32 + (((uint64_t)m.p << 32) | (uint32_t)acc[r]);
    }
    if (n & 4) {
#pragma unroll
      for (int u = 0; u < 4; ++u) step(u);
      pa += 4 * C;
      pw += 8;
    }
    if (n & 2) {
#pragma unroll
      for (int u = 0; u < 2; ++u) step(u);
      pa += 2 * C;
      pw += 4;
    }
    if (n & 1) step(0);
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const uint32_t h = (uint32_t)(acc[r] >> 32);  // < 15 2^28 + 2^21 < 2 p
      const uint32_t v = redc(((uint64_t)rs_umin(h, h - m.p) << 32) | (uint32_t)acc[r], m.p, m.pinv);
      const uint32_t s = v + __shfl_xor_sync(0xffffffffu, v * sg + off, 1);  // < 2 p
      const uint32_t z = rs_umin(s, s - m.p);
      if constexpr (COL) {
        pc[r] = z;
      } else {
#pragma unroll
        for (int q = 0; q < C; q += 8)
          if (q == 8 * b) P[q + r] = z;
      }
    }
    pc += 8;
  }
  if constexpr (COL) {
#pragma unroll
    for (int r = 0; r < C; ++r) P[r] = col[r];
  }
}

// Row k of the staged coefficients, k < 2 g1_half_rows(dx); qn[t] = q^{-C(t,2)}.
// From 8 limbs the coefficients' products are summed before one reduction (for
// 1 to 4 limbs that, or a choice inside the loop, costs 1 to 4% of the whole
// kernel: hence a function of its own).  When long ones fill less than 40% of
// the padded rows they are taken from a list of those that exist (column j's
// start at smeta[j].x - smeta[0].x), so that a warp does not walk the limbs of
// its few lanes that have one.  G1, us: 23,980 (pair, prime) items of 55 and 10
// coefficients of 64 limbs 478 -> 343 (456 with the padded rows alone); 40,000
// of 136 and 16 2,120 -> 1,868; 10,280 of those with 16 limbs 454 -> 442.
template <int C>
__device__ __noinline__ void stage_long(int32_t *sa, const int2 *smeta, int deg, int dx, int nc,
                                        const uint32_t *limbs, int stride, int L,
                                        const uint32_t *V, const uint32_t *qn, const ModP m) {
  const int n = 2 * g1_half_rows(dx) * C, odd = g1_odd_offset(dx, C);
  if (5 * nc >= 2 * n) {
    for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
      const int k = idx / C, r = idx - k * C, j = deg - r;
      int32_t v = 0;
      if (j >= 0 && k <= smeta[j].y)
        v = signed_rep(mmul(reduce_long(limbs + ((size_t)k * stride + j) * L, L, V, m), qn[k], m), m.p);
      sa[(k & 1) * odd + (k >> 1) * C + r] = v;
    }
    return;
  }
  for (int idx = threadIdx.x; idx < n; idx += blockDim.x) sa[(idx / C & 1) * odd + (idx / C >> 1) * C + idx % C] = 0;
  __syncthreads();
  for (int e = threadIdx.x; e < nc; e += blockDim.x) {
    const int at = smeta[0].x + e;
    int j = 0, hi = deg;  // the last column that starts at or before e: it has coefficients
    while (j < hi) {
      const int mid = (j + hi + 1) >> 1;
      if (smeta[mid].x <= at)
        j = mid;
      else
        hi = mid - 1;
    }
    const int k = at - smeta[j].x;
    const uint32_t c = reduce_long(limbs + ((size_t)k * stride + j) * L, L, V, m);
    sa[(k & 1) * odd + (k >> 1) * C + deg - j] = signed_rep(mmul(c, qn[k], m), m.p);
  }
}

template <int C>
__device__ __forceinline__ void stage_chirp(int32_t *sa, const int2 *smeta, int deg, int dx, int nc,
                                            const uint32_t *limbs, int stride, int L,
                                            const uint32_t *V, const uint32_t *qn, const ModP &m) {
  if (L >= 8) {
    stage_long<C>(sa, smeta, deg, dx, nc, limbs, stride, L, V, qn, m);
    return;
  }
  const int n = 2 * g1_half_rows(dx) * C, odd = g1_odd_offset(dx, C);
  for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
    const int k = idx / C, r = idx - k * C, j = deg - r;
    int32_t v = 0;
    if (j >= 0 && k <= smeta[j].y)
      v = signed_rep(mmul(reduce_coef(limbs + ((size_t)k * stride + j) * L, L, V, m), qn[k], m), m.p);
    sa[(k & 1) * odd + (k >> 1) * C + r] = v;
  }
}

template <int C, bool COL>
__global__ void __launch_bounds__(128, COL ? RS_G1_MINB : 2) g1_kernel(G1Args a) {
  extern __shared__ __align__(16) uint32_t sm[];
  __shared__ int s_tile;
  bool first = true;
  for (;;) {
    int t;
    if (a.persistent) {
      if (threadIdx.x == 0) s_tile = atomicAdd(a.counter, 1);
      __syncthreads();
      t = s_tile;
    } else {
      t = first ? (int)blockIdx.x : a.ntiles;
    }
    first = false;
    if (t >= a.ntiles) return;

    const Tile tl = a.tiles[t];
    const PairDesc pd = a.pairs[tl.pair];
    const ModP m = a.mods[tl.prime];
    const uint32_t *V = a.vtab + (size_t)tl.prime * RS_VT_STRIDE;
    const int nmeta = pd.my + pd.ny + 2;
    const int dxm = max(pd.mxf, pd.mxg);
    int2 *smeta = reinterpret_cast<int2 *>(sm);
    int32_t *ssteps = reinterpret_cast<int32_t *>(sm) + 2 * nmeta;  // rows per parity of each block of 8 columns
    int32_t *saf = reinterpret_cast<int32_t *>(sm) + ((2 * nmeta + 2 * (C / 8) + 7) & ~7);  // 32-byte aligned
    int32_t *sag = saf + ((g1_poly_words(pd.mxf, C) + 7) & ~7);
    int32_t *swin = sag + g1_poly_words(pd.mxg, C);
    uint32_t *scol = reinterpret_cast<uint32_t *>(swin) + (blockDim.x >> 1) + dxm + 2 + threadIdx.x * (C + 1);  // odd stride; with COL
    const size_t tb = (size_t)tl.prime * a.tstride;

    for (int i = threadIdx.x; i < nmeta; i += blockDim.x) smeta[i] = a.meta[pd.meta_off + i];
    __syncthreads();
    stage_chirp<C>(saf, smeta, pd.my, pd.mxf, pd.fnc, a.limbs + pd.f_off, pd.fstride, pd.Lf, V, a.qn + tb, m);
    stage_chirp<C>(sag, smeta + pd.my + 1, pd.ny, pd.mxg, pd.gnc, a.limbs + pd.g_off, pd.gstride, pd.Lg, V,
                   a.qn + tb, m);
    for (int i = threadIdx.x; i < 2 * (C / 8); i += blockDim.x) {
      const int w = i / (C / 8), top = (w ? pd.ny : pd.my) - 8 * (i - w * (C / 8));
      int k = -2;
      for (int r = 0; r < 8; ++r)
        if (top - r >= 0) k = max(k, smeta[w * (pd.my + 1) + top - r].y);
      ssteps[i] = (k >> 1) + 1;  // x-degree -1 (a zero coefficient): no row
    }
    __syncthreads();

    if (tl.x0 == 0 && threadIdx.x == 0) {  // unlucky prime: a leading coefficient vanishes mod p
      bool zf = true, zg = true;
      for (int k = 0; k <= pd.mxf; ++k) zf = zf && saf[(k & 1) * g1_odd_offset(pd.mxf, C) + (k >> 1) * C] == 0;
      for (int k = 0; k <= pd.mxg; ++k) zg = zg && sag[(k & 1) * g1_odd_offset(pd.mxg, C) + (k >> 1) * C] == 0;
      if (zf || zg) atomicAdd(a.stats + ST_UNLUCKY_PRIMES, 1ull);
    }

    // The work item's point pairs [x0, x0 + n) in chunks of blockDim / 2: the
    // staged coefficients serve every chunk, only the window is reloaded.
    const int ti = (int)threadIdx.x >> 1, par = (int)threadIdx.x & 1;
    const int half = (int)(blockDim.x >> 1);
    for (int cx = tl.x0; cx < tl.x0 + tl.n; cx += half) {
      const int nn = min(half, tl.x0 + tl.n - cx);
      for (int t = threadIdx.x; t < half + dxm + 2; t += blockDim.x) swin[t] = a.qc[tb + cx + t];
      __syncthreads();
      uint32_t unlucky = 0u, degen = 0u;
      const int i = cx + ti;  // point pair: this thread's image is at (-1)^par q^i
      // every thread evaluates (the shuffles need the whole warp); only the
      // threads of the chunk's pairs run the remainder sequence
      uint32_t A[C], B[C];
      eval_chirp<C, COL>(A, saf + par * g1_odd_offset(pd.mxf, C), ssteps, swin + ti + par, scol, par, m);
      eval_chirp<C, COL>(B, sag + par * g1_odd_offset(pd.mxg, C), ssteps + C / 8, swin + ti + par, scol, par, m);
      if (ti < nn) {
        unlucky = (A[0] == 0u || B[0] == 0u) ? 1u : 0u;
        Prs s;
        s.a = pd.my;
        s.b = pd.ny;
        s.num = s.den = s.Q = m.r1;
        s.eprev = max(min(pd.my, pd.ny) - 1, 0);
        s.sign = (uint32_t)(par & (pd.my + pd.ny));  // A and B are negated in odd lanes
        s.degen = 0u;
        prs_run<C>(A, B, s, m);
        // the chirp factor left out of the coefficients (reloaded: no register held through the sequence)
        s.num = mmul(s.num, mpow(a.qn[tb + i], (uint32_t)(pd.my + pd.ny), m), m);
        while (s.eprev > 0) {
          s.den = mmul(s.den, s.Q, m);
          --s.eprev;
        }
        const size_t idx = (size_t)pd.img_off + (size_t)tl.prime * pd.NI + 2 * i + par;
        a.num[idx] = s.sign ? mneg(s.num, m.p) : s.num;
        a.den[idx] = s.den;
        degen = s.degen;
      }
      const unsigned bu = __ballot_sync(0xffffffffu, unlucky);
      const unsigned bd = __ballot_sync(0xffffffffu, degen);
      if ((threadIdx.x & 31) == 0) {
        if (bu) atomicAdd(a.stats + ST_UNLUCKY_POINTS, (unsigned long long)__popc(bu));
        if (bd) atomicAdd(a.stats + ST_DEGENERATE, (unsigned long long)__popc(bd));
      }
      __syncthreads();  // the next chunk reloads the window (the next item restages everything)
    }
  }
}

}  // namespace

#ifndef RS_G1_CAP
#error "compile this file once per register capacity with -DRS_G1_CAP=<8..72>"
#endif
#define RS_CAT2(a, b) a##b
#define RS_CAT(a, b) RS_CAT2(a, b)

cudaError_t RS_CAT(rs_g1_launch_, RS_G1_CAP)(bool col, int threads, int blocks, size_t smem, const G1Args &a,
                                            cudaStream_t s) {
  if (col)
    g1_kernel<RS_G1_CAP, true><<<blocks, threads, smem, s>>>(a);
  else
    g1_kernel<RS_G1_CAP, false><<<blocks, threads, smem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t RS_CAT(rs_g1_prepare_, RS_G1_CAP)(bool col, int threads, size_t smem, int *mb) {
  // The attribute is per kernel, not per launch: always allow the largest
  // staging any plan may request so that batches prepared earlier with more
  // shared memory keep working.
  const void *k = col ? (const void *)g1_kernel<RS_G1_CAP, true> : (const void *)g1_kernel<RS_G1_CAP, false>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, RS_G1_MAX_SMEM_BYTES);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(mb, k, threads, smem);
}
