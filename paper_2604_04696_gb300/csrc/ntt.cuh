// Negacyclic NTT, its inverse and the gadget digit decomposition (Dcp) on one
// CTA, for the ciphertext-tree kernels of ColTor and ExpandQuery (GPIR paper
// Sec. 2.4.1 for the NTT, Sec. 2.5.1 for the Inverse NTT -> Dcp -> Forward
// NTT -> multiply-accumulate chain they share).
//
// Transform: A_s = sum_j a_j psi^((2s+1) j) mod q, psi = g^((q-1)/2N) with g
// the smallest generator of Z_q^* (the NTT form RowSel's data is in), slots in
// natural order. The butterfly networks are the merged-twist Cooley-Tukey
// (forward, natural -> bit-reversed) and Gentleman-Sande (inverse,
// bit-reversed -> natural) networks of Longa and Naehrig ("Speeding up the
// Number Theoretic Transform for Faster Ideal Lattice-Based Cryptography",
// CANS 2016), with twiddles psi^brv(k) and psi^-brv(k).
//
// Arithmetic: Harvey's lazy butterflies ("Faster arithmetic for
// number-theoretic transforms", J. Symb. Comp. 2014) with Shoup products:
// a * w mod q for a fixed w is a*w - floor(a * w' / 2^32) * q with
// w' = floor(w 2^32 / q), a value in [0, 2q) for any 32-bit a. The transforms
// let values grow as far as 32 bits allow (q < 2^28, so 16q <= 2^32), with
// every bound tracked at compile time:
//   - forward: a level adds 2q; the upper operand of a butterfly is brought
//     below 8q only where the sum could pass 16q. From inputs below 2q that
//     is at levels 7 and 11 of 12: one conditional subtraction per point of a
//     4096-point transform. Outputs are below 16q;
//   - inverse: sums double, products are below 2q; within a radix-8 round the
//     bounds of the 8 values are 16, 8, 4, 4, 2, 2, 2, 2 (times q), and the
//     four larger ones are brought below 2q at its end.
// A conditional subtraction x >= c ? x - c : x is min(x, x - c) on unsigned
// values.
//
// GPU mapping. A polynomial of one limb belongs to a CTA of N/8 threads (the
// kernels run one CTA per limb of a tree node, the limbs of a node in one
// thread-block cluster). The digit polynomials of a node go through the
// forward transform together, so a round's twiddles are loaded once for all of
// them and they share its barrier; a round's twiddles are loaded before the
// barrier it starts with. Thread b of the CTA owns the 8 points
// b + (N/8) e, e = 0..7, in registers on both ends of a transform, so the
// transforms chain with the coefficient-wise Dcp and the slot-wise
// multiply-accumulate without a trip through memory:
//   - forward: the first radix-8 round (levels 0-2) works on exactly the
//     owned coefficients; the last radix-8 round works on 8 consecutive
//     bit-reversed positions 8i+k, and with i = brv(b) those hold the owned
//     slots b + (N/8) brv3(k), so no bit-reversal pass is needed;
//   - inverse: the mirror image (first round on the owned slots at positions
//     8 brv(b) + k, last round on the owned coefficients).
// Middle rounds go through shared memory: one load of 8 values, three levels
// of butterflies in registers, one store, one barrier. N is a template
// parameter, so every round's geometry is a compile-time constant.
//
// Shared-memory layout: position x lives at word pad(x) = x + 4 (x >> 9) of a
// buffer of padn(N) words. Every set of every round has the form
// base + k u with base = i 2^R u + o, o < u, and for those
// pad(base + k u) = pad(base) + k u + 4 (k u >> 9): one address per set, the
// rest are immediate offsets. Four pad words per 512 keep groups of 4
// positions 16-byte aligned, so the bit-reversed rounds (8 consecutive
// positions per thread) move two 16-byte words, and with the thread-to-set map
// of the 64i + o + 8k round below every access of every round at N = 4096 is
// free of bank conflicts (8 consecutive threads of a bit-reversed round sit
// 512 positions apart, which the pad spreads over all banks).
#pragma once

#include <stdint.h>

#include "common.cuh"
#include "internal.h"

namespace gpir {
namespace ntt {

constexpr uint32_t MAX_N = 4096;
constexpr uint32_t MIN_N = 16;
constexpr int MIN_LOGN = 4, MAX_LOGN = 12;
constexpr uint32_t MAX_LIMBS = 2;
constexpr int LOG_BASE = 22;              // gadget base z = 2^22 (the paper's)

// Threads of a CTA that owns one limb polynomial (N/8 of them do transform
// work, at least a warp), and the CTAs per SM that its 64 registers a thread
// allow.
template <int LOGN>
__host__ __device__ constexpr int threads() { return LOGN >= 8 ? 1 << (LOGN - 3) : 32; }
template <int LOGN>
__host__ __device__ constexpr int ctas_per_sm() { return 1024 / threads<LOGN>() > 16 ? 16 : 1024 / threads<LOGN>(); }
// Digit polynomials a node transforms together: the most that L 28-bit limbs
// need. Smaller moduli need fewer digits; the absent ones are zero.
template <int L>
__host__ __device__ constexpr int digits() { return L == 1 ? 2 : 3; }

struct Limb {
  const uint2 *fw;        // [N]  (psi^brv(k), Shoup quotient)
  const uint2 *iv;        // [N]  (psi^-brv(k), Shoup quotient)
  const uint2 *fw_last;   // [N/8][8]: the twiddles of the last forward round of thread b, in thread order
  const uint2 *iv_first;  // [N/8][8]: the twiddles of the first inverse round of thread b, in thread order
  const uint2 *mono;      // [2N] (psi^-e, Shoup quotient): slot s of NTT(X^-m) is psi^-((2s+1) m mod 2N)
  uint2 fw8[8];           // fw[1..7] at 1..7: the first forward round, the same for every thread
  uint2 iv8[8];           // iv[4..7], iv[2..3], iv[1] / N at 0..6: the last inverse round with its scaling
  uint2 n_inv;            // 1 / N mod q and its Shoup quotient
  uint2 r32;              // 2^32 mod q and its Shoup quotient
  uint32_t q, one_s;      // one_s = floor(2^32 / q): the Shoup quotient of 1
  uint32_t q2, pad;       // 2q: kept as a value of its own, so that u - t + 2q stays one three-operand addition
  uint32_t digit_add[3];  // added to the masked digit field i: minus its offset plus a multiple of q, >= 0
};

struct Ring {
  uint32_t L, N, logn, ell;
  uint64_t half_Q;        // floor(Q / 2), Q = prod q_l (< 2^56)
  uint64_t off_pos, off_neg;   // O and O - Q, O = sum_{k < ell-1} 2^21 2^(22 k): y = centred x + O
  uint32_t digit_mask[3]; // field i of y: 22 bits below the top digit, all bits for it, 0 past it
  uint32_t crt_add;       // multiple of q1, >= q0
  uint2 q0_inv;           // q0^-1 mod q1 and its Shoup quotient (L = 2)
  Limb limb[MAX_LIMBS];
};

__host__ __device__ constexpr uint32_t padn(uint32_t n) { return n + 4 * (n >> 9); }
__host__ __device__ constexpr uint32_t pad(uint32_t x) { return x + 4 * (x >> 9); }
__device__ __forceinline__ uint32_t brev(uint32_t x, uint32_t bits) { return bits ? __brev(x) >> (32 - bits) : 0u; }

__device__ __forceinline__ uint32_t csub(uint32_t x, uint32_t c) { return min(x, x - c); }
__device__ __forceinline__ uint32_t shoup_lazy(uint32_t a, uint2 w, uint32_t q) {
  return a * w.x - __umulhi(a, w.y) * q;
}
__device__ __forceinline__ uint32_t shoup(uint32_t a, uint2 w, uint32_t q) { return csub(shoup_lazy(a, w, q), q); }
// Any 32-bit x to [0, 2q): Shoup's product by 1.
__device__ __forceinline__ uint32_t red32(uint32_t x, const Limb &T) { return x - __umulhi(x, T.one_s) * T.q; }
// Any 64-bit x to [0, 4q): hi 2^32 + lo by two Shoup products, of 2^32 and of
// 1, whose quotients are summed before the one product by q.
__device__ __forceinline__ uint32_t red64(uint64_t x, const Limb &T) {
  const uint32_t hi = (uint32_t)(x >> 32), lo = (uint32_t)x;
  return hi * T.r32.x + lo - (__umulhi(hi, T.r32.y) + __umulhi(lo, T.one_s)) * T.q;
}
// [0, 4q) to [0, q).
__device__ __forceinline__ uint32_t csub4(uint32_t x, uint32_t q) { return csub(csub(x, 2 * q), q); }

__device__ __forceinline__ uint4 ld4(const uint2 *p) { return __ldg(reinterpret_cast<const uint4 *>(p)); }
__device__ __forceinline__ uint2 ld2(const uint2 *p) { return __ldg(p); }

// Bound (in units of q) of a forward transform's values before level l, from
// inputs below 2q: a level adds 2 and starts at 8 again where that would pass
// 16 (levels 7 and 11). Closed forms, so that unrolled code folds them.
__host__ __device__ constexpr int fwd_bound(int l) { return l <= 7 ? 2 + 2 * l : l <= 11 ? 2 * l - 6 : 10; }
// Bound of value k of an inverse round before its level r, from values below
// 2q: products are below 2q and sums double, so it counts the levels since
// the last one that multiplied (the highest set bit of k below bit r).
__host__ __device__ constexpr int inv_bound(int k, int r) {
  return r == 0 || (k >> (r - 1)) & 1 ? 2 : r == 1 || (k >> (r - 2)) & 1 ? 4 : r == 2 || (k >> (r - 3)) & 1 ? 8 : 16;
}

// R forward levels (Cooley-Tukey: x, y -> x + w y, x - w y), the first of them
// level LVL of the transform, on P polynomials. w[2^r - 1 + j] is the twiddle
// of the pairs k with k >> (R - r) = j at level r.
template <int R, int LVL, int P>
__device__ __forceinline__ void fwd_levels(uint32_t (&v)[P][8], const uint2 (&w)[7], const Limb &T) {
  const uint32_t q = T.q, q2 = T.q2;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int span = 1 << (R - 1 - r);
#pragma unroll
    for (int k = 0; k < (1 << R); ++k) {
      if (k & span) continue;
      const uint2 tw = w[(1 << r) - 1 + (k >> (R - r))];
#pragma unroll
      for (int p = 0; p < P; ++p) {
        const uint32_t t = shoup_lazy(v[p][k + span], tw, q);
        const uint32_t u = fwd_bound(LVL + r) + 2 > 16 ? csub(v[p][k], 8 * q) : v[p][k];
        v[p][k] = u + t;
        v[p][k + span] = u - t + q2;
      }
    }
  }
}

// R inverse levels (Gentleman-Sande: x, y -> x + y, w (x - y)). Level r pairs
// k with k + 2^r; w holds level 0's 2^(R-1) twiddles, then level 1's, ...
// LAST: the transform's last round (R = 3), whose values are scaled by 1/N and
// reduced below q (the twiddle of its last level includes the 1/N); otherwise
// values end below 2q.
template <int R, bool LAST, int P>
__device__ __forceinline__ void inv_levels(uint32_t (&v)[P][8], const uint2 (&w)[7], const Limb &T) {
  const uint32_t q = T.q, q2 = T.q2;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int span = 1 << r, first = (1 << R) - (1 << (R - r));
#pragma unroll
    for (int k = 0; k < (1 << R); ++k) {
      if (k & span) continue;
      const uint2 tw = w[first + (k >> (r + 1))];
#pragma unroll
      for (int p = 0; p < P; ++p) {
        const uint32_t x = v[p][k], y = v[p][k + span];
        v[p][k] = x + y;
        v[p][k + span] = shoup_lazy(x - y + (inv_bound(k + span, r) == 2 ? q2 : inv_bound(k + span, r) / 2 * q2), tw, q);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < (1 << R); ++k) {
    const int bound = inv_bound(k, R);
#pragma unroll
    for (int p = 0; p < P; ++p) {
      if (LAST) v[p][k] = csub(k < (1 << (R - 1)) ? shoup_lazy(v[p][k], T.n_inv, q) : v[p][k], q);
      else if (bound > 4) v[p][k] = red32(v[p][k], T);
      else if (bound > 2) v[p][k] = csub(v[p][k], q2);
    }
  }
}

// Twiddles of a forward round of R levels on the set of group i, M0 = 2^l0
// groups at its first level l0.
template <int R, uint32_t M0>
__device__ __forceinline__ void fwd_twiddles(uint2 (&w)[7], const uint2 *fw, uint32_t i) {
  w[0] = ld2(fw + i + M0);
  if constexpr (R >= 2) {
    const uint4 b = ld4(fw + 2 * i + 2 * M0);
    w[1] = make_uint2(b.x, b.y);
    w[2] = make_uint2(b.z, b.w);
  }
  if constexpr (R == 3) {
    const uint4 c = ld4(fw + 4 * i + 4 * M0), d = ld4(fw + 4 * i + 4 * M0 + 2);
    w[3] = make_uint2(c.x, c.y);
    w[4] = make_uint2(c.z, c.w);
    w[5] = make_uint2(d.x, d.y);
    w[6] = make_uint2(d.z, d.w);
  }
}

// Twiddles of an inverse round of R levels on the set of group i, H0 = N/(2 t0).
template <int R, uint32_t H0>
__device__ __forceinline__ void inv_twiddles(uint2 (&w)[7], const uint2 *iv, uint32_t i) {
  if constexpr (R == 3) {
    const uint4 a = ld4(iv + 4 * i + H0), b = ld4(iv + 4 * i + H0 + 2);
    w[0] = make_uint2(a.x, a.y);
    w[1] = make_uint2(a.z, a.w);
    w[2] = make_uint2(b.x, b.y);
    w[3] = make_uint2(b.z, b.w);
  }
  if constexpr (R >= 2) {
    const uint4 c = ld4(iv + 2 * i + H0 / (R == 3 ? 2 : 1));
    w[R == 3 ? 4 : 0] = make_uint2(c.x, c.y);
    w[R == 3 ? 5 : 1] = make_uint2(c.z, c.w);
  }
  w[R == 3 ? 6 : R == 2 ? 2 : 0] = ld2(iv + i + H0 / (1 << (R - 1)));
}

// The bit-reversed rounds (the last forward round and the first inverse round,
// set i = brv(b)) touch 7/8 of the twiddle table, scattered over the threads of
// a warp. Their twiddles are also stored per thread, in thread order (64 bytes
// each, see ring_tables.cu), so that these loads are contiguous across a warp:
//   fw_last[b]  = W[N/8 + i], W[N/4 + 2i], W[N/4 + 2i + 1], -, W[N/2 + 4i + 0..3]
//   iv_first[b] = V[N/2 + 4i + 0..3], V[N/4 + 2i], V[N/4 + 2i + 1], V[N/8 + i], -
__device__ __forceinline__ void thread_twiddles(uint2 (&w)[7], const uint2 *t, bool forward) {
  const uint4 a = ld4(t), b = ld4(t + 2), c = ld4(t + 4), d = ld4(t + 6);
  w[0] = make_uint2(a.x, a.y);
  w[1] = make_uint2(a.z, a.w);
  w[2] = make_uint2(b.x, b.y);
  if (forward) {
    w[3] = make_uint2(c.x, c.y);
    w[4] = make_uint2(c.z, c.w);
    w[5] = make_uint2(d.x, d.y);
    w[6] = make_uint2(d.z, d.w);
  } else {
    w[3] = make_uint2(b.z, b.w);
    w[4] = make_uint2(c.x, c.y);
    w[5] = make_uint2(c.z, c.w);
    w[6] = make_uint2(d.x, d.y);
  }
}

// Levels of the next middle round when LEFT levels remain (4 -> 2 + 2, so that
// no round is a lone radix-2 when it can be avoided).
template <int LEFT>
__host__ __device__ constexpr int middle_levels() { return LEFT == 4 ? 2 : (LEFT < 3 ? LEFT : 3); }

// Thread-to-set map of a middle round (run by the threads b < N/8, each
// taking sets b, b + N/8, ...): set sb -> (group i, offset o), INNER = the
// offset range (u forward, t0 inverse). The radix-8 round whose sets are
// 64i + o + 8k (INNER = 8) takes i = warp + (N/256) ((sb >> 3) & 3), which
// spreads a warp over 4 groups 16 apart; every other round maps
// sb = i INNER + o.
template <int R, uint32_t INNER, uint32_t N>
__device__ __forceinline__ void set_of(uint32_t sb, uint32_t &i, uint32_t &o) {
  if constexpr (R == 3 && INNER == 8 && N >= 256) {
    o = sb & 7;
    i = (sb >> 5) + (N >> 8) * ((sb >> 3) & 3);
  } else {
    i = sb / INNER;
    o = sb % INNER;
  }
}

// Levels still to do when the bit-reversed round (if the ring is large enough
// to have one) begins.
template <int LOGN>
__host__ __device__ constexpr int middle_end() { return LOGN >= 6 ? LOGN - 3 : LOGN; }

// Twiddles of thread b's round that starts at forward level LVL, where each
// thread has one set in it (otherwise the round loads them itself).
template <int LOGN, int LVL>
__device__ __forceinline__ void fwd_next_twiddles(uint2 (&w)[7], const Limb &T, uint32_t b) {
  constexpr int LEFT = middle_end<LOGN>() - LVL;
  if constexpr (LEFT > 0) {
    if constexpr (middle_levels<LEFT>() == 3) {
      uint32_t i, o;
      set_of<3, ((1u << LOGN) >> (LVL + 3)), (1u << LOGN)>(b, i, o);
      fwd_twiddles<3, 1u << LVL>(w, T.fw, i);
    }
  } else if constexpr (LOGN >= 6) {
    thread_twiddles(w, T.fw_last + 8 * b, true);
  }
}

// The same for the inverse round at level G.
template <int LOGN, int G>
__device__ __forceinline__ void inv_next_twiddles(uint2 (&w)[7], const Limb &T, uint32_t b) {
  constexpr int LEFT = middle_end<LOGN>() - G;
  if constexpr (LEFT > 0) {
    if constexpr (middle_levels<LEFT>() == 3) {
      uint32_t i, o;
      set_of<3, (1u << G), (1u << LOGN)>(b, i, o);
      inv_twiddles<3, (1u << LOGN) / (2u << G)>(w, T.iv, i);
    }
  }
}

template <int LOGN, int R, int LVL, int P>
__device__ __forceinline__ void fwd_middle(uint32_t *const (&buf)[P], uint2 (&w)[7], const Limb &T, uint32_t b) {
  constexpr uint32_t N = 1u << LOGN, S = N >> 3, M0 = 1u << LVL, U = N >> (LVL + R);
#pragma unroll
  for (uint32_t t = 0; t < (N >> R) / S; ++t) {
    uint32_t i, o;
    set_of<R, U, N>(b + t * S, i, o);
    const uint32_t base = pad((i << R) * U + o);
    if constexpr (R < 3) fwd_twiddles<R, M0>(w, T.fw, i);
    uint32_t v[P][8];
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (uint32_t k = 0; k < (1u << R); ++k) v[p][k] = buf[p][base + pad(k * U)];
    fwd_levels<R, LVL, P>(v, w, T);
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (uint32_t k = 0; k < (1u << R); ++k) buf[p][base + pad(k * U)] = v[p][k];
  }
}

template <int LOGN, int R, int G>
__device__ __forceinline__ void inv_middle(uint32_t *buf, uint2 (&w)[7], const Limb &T, uint32_t b) {
  constexpr uint32_t N = 1u << LOGN, S = N >> 3, T0 = 1u << G;
#pragma unroll
  for (uint32_t t = 0; t < (N >> R) / S; ++t) {
    uint32_t i, o;
    set_of<R, T0, N>(b + t * S, i, o);
    uint32_t *p = buf + pad((i << R) * T0 + o);
    if constexpr (R < 3) inv_twiddles<R, N / (2 * T0)>(w, T.iv, i);
    uint32_t v[1][8];
#pragma unroll
    for (uint32_t k = 0; k < (1u << R); ++k) v[0][k] = p[pad(k * T0)];
    inv_levels<R, false, 1>(v, w, T);
#pragma unroll
    for (uint32_t k = 0; k < (1u << R); ++k) p[pad(k * T0)] = v[0][k];
  }
}

// The rounds from level LVL (G) to the bit-reversed (last) one; w holds the
// first one's twiddles on entry and the next round's on return.
template <int LOGN, int LVL, int P>
__device__ __forceinline__ void fwd_middles(uint32_t *const (&buf)[P], uint2 (&w)[7], const Limb &T, uint32_t b,
                                            bool act) {
  if constexpr (LVL < middle_end<LOGN>()) {
    constexpr int R = middle_levels<middle_end<LOGN>() - LVL>();
    if (act) {
      fwd_middle<LOGN, R, LVL, P>(buf, w, T, b);
      fwd_next_twiddles<LOGN, LVL + R>(w, T, b);
    }
    __syncthreads();
    fwd_middles<LOGN, LVL + R, P>(buf, w, T, b, act);
  }
}

template <int LOGN, int G>
__device__ __forceinline__ void inv_middles(uint32_t *buf, uint2 (&w)[7], const Limb &T, uint32_t b, bool act) {
  if constexpr (G < middle_end<LOGN>()) {
    constexpr int R = middle_levels<middle_end<LOGN>() - G>();
    if (act) {
      inv_middle<LOGN, R, G>(buf, w, T, b);
      inv_next_twiddles<LOGN, G + R>(w, T, b);
    }
    __syncthreads();
    inv_middles<LOGN, G + R>(buf, w, T, b, act);
  }
}

// Forward NTT of P polynomials of one limb (one padded buffer of padn(N) words
// each). In: v[p][k] = coefficient b + (N/8) k, values < 2q. Out: v[p][e] =
// slot b + (N/8) e, values in [0, 16q) (lazy: congruent mod q, not reduced).
// Every thread of the CTA must call it (it holds __syncthreads); act = b < N/8.
// Before its first barrier a thread writes only the positions b + (N/8) k of
// the buffers; after its last one it reads only the positions 8 brv(b) + k.
// Those are also the positions that inverse() writes before its first barrier,
// in the same thread, so an inverse() may follow with no barrier in between
// (ExpandQuery's loop over nodes with one limb); any other use of the buffers
// waits for the next barrier of the CTA.
template <int LOGN, int P>
__device__ __forceinline__ void forward(uint32_t (&v)[P][8], uint32_t *const (&buf)[P], const Limb &T, uint32_t b,
                                        bool act) {
  constexpr uint32_t N = 1u << LOGN, S = N >> 3;
  uint2 w[7];
  if (act) {
#pragma unroll
    for (int k = 0; k < 7; ++k) w[k] = T.fw8[k + 1];
    fwd_levels<3, 0, P>(v, w, T);
    const uint32_t base = pad(b);
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (uint32_t k = 0; k < 8; ++k) buf[p][base + pad(k * S)] = v[p][k];
    fwd_next_twiddles<LOGN, 3>(w, T, b);
  }
  __syncthreads();
  fwd_middles<LOGN, 3, P>(buf, w, T, b, act);
  if (!act) return;
  if constexpr (LOGN >= 6) {
    const uint32_t base = pad(8 * brev(b, LOGN - 3));
#pragma unroll
    for (int p = 0; p < P; ++p) {
      const uint4 x = *reinterpret_cast<const uint4 *>(buf[p] + base);
      const uint4 y = *reinterpret_cast<const uint4 *>(buf[p] + base + 4);
      v[p][0] = x.x, v[p][1] = x.y, v[p][2] = x.z, v[p][3] = x.w;
      v[p][4] = y.x, v[p][5] = y.y, v[p][6] = y.z, v[p][7] = y.w;
    }
    fwd_levels<3, LOGN - 3, P>(v, w, T);
#pragma unroll
    for (int p = 0; p < P; ++p) {
      // position 8i + k holds slot (N/8) brv3(k) + b
      const uint32_t t1 = v[p][1], t3 = v[p][3];
      v[p][1] = v[p][4], v[p][4] = t1;
      v[p][3] = v[p][6], v[p][6] = t3;
    }
  } else {
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (uint32_t e = 0; e < 8; ++e) v[p][e] = buf[p][pad(brev(b + e * S, LOGN))];
  }
}

// Twiddles of the first inverse round, which a kernel loads before it has the
// values.
template <int LOGN>
__device__ __forceinline__ void inv_first_twiddles(uint2 (&w)[7], const Limb &T, uint32_t b) {
  if constexpr (LOGN >= 6) thread_twiddles(w, T.iv_first + 8 * b, false);
  else inv_twiddles<3, (1u << LOGN) / 2>(w, T.iv, brev(b, LOGN - 3));
}

// Inverse NTT of one polynomial of one limb. In: v[e] = slot b + (N/8) e,
// values < 2q, and w from inv_first_twiddles. Out: v[k] = coefficient
// b + (N/8) k, below q. Before its first barrier a thread writes only the
// positions 8 brv(b) + k of the buffer; after its last one it reads only the
// positions b + (N/8) k.
template <int LOGN>
__device__ __forceinline__ void inverse(uint32_t (&v)[1][8], uint32_t *buf, uint2 (&w)[7], const Limb &T,
                                        uint32_t b, bool act) {
  constexpr uint32_t N = 1u << LOGN, S = N >> 3;
  if (act) {
    // position 8i + k, i = brv(b), holds slot (N/8) brv3(k) + b
    const uint32_t t1 = v[0][1], t3 = v[0][3];
    v[0][1] = v[0][4], v[0][4] = t1;
    v[0][3] = v[0][6], v[0][6] = t3;
    inv_levels<3, false, 1>(v, w, T);
    uint4 *p = reinterpret_cast<uint4 *>(buf + pad(8 * brev(b, LOGN - 3)));
    p[0] = make_uint4(v[0][0], v[0][1], v[0][2], v[0][3]);
    p[1] = make_uint4(v[0][4], v[0][5], v[0][6], v[0][7]);
    inv_next_twiddles<LOGN, 3>(w, T, b);
  }
  __syncthreads();
  inv_middles<LOGN, 3>(buf, w, T, b, act);
  if (!act) return;
  const uint32_t base = pad(b);
#pragma unroll
  for (uint32_t k = 0; k < 8; ++k) v[0][k] = buf[base + pad(k * S)];
  if constexpr (LOGN >= 6) {
#pragma unroll
    for (int k = 0; k < 7; ++k) w[k] = T.iv8[k];
    inv_levels<3, true, 1>(v, w, T);
  } else {
#pragma unroll
    for (uint32_t k = 0; k < 8; ++k) v[0][k] = shoup(v[0][k], T.n_inv, T.q);
  }
}

// Dcp: y = x + O for the centred CRT value x in (-Q/2, Q/2] of one coefficient
// with residues (r0 mod q0, r1 mod q1) (Garner for L = 2), where
// O = sum_{k < ell-1} (z/2) z^k. The balanced base-z digits of x are then
// plain fields of y: d_k = ((y >> 22k) mod z) - z/2 for k < ell - 1, and the
// top digit is y >> 22 (ell - 1) (arithmetic shift; its low 32 bits hold it).
// d[i] is digit i mod q, below 2q.
template <int L>
__device__ __forceinline__ void dcp_digits(const Ring &R, const Limb &T, uint32_t r0, uint32_t r1,
                                           uint32_t (&d)[digits<L>()]) {
  uint64_t x = r0;
  if constexpr (L > 1) {
    const uint32_t k = shoup(r1 + R.crt_add - r0, R.q0_inv, R.limb[1].q);
    x += (uint64_t)R.limb[0].q * k;
  }
  const uint64_t y = x + (x > R.half_Q ? R.off_neg : R.off_pos);
#pragma unroll
  for (int i = 0; i < digits<L>(); ++i)
    d[i] = ((uint32_t)((int64_t)y >> (LOG_BASE * i)) & R.digit_mask[i]) + T.digit_add[i];
}

// Programmatic dependent launch: a stage's grid starts while the stage before
// it finishes. It may read only what no earlier stage writes until it has
// waited (the wait returns at once when the grid was launched without the
// attribute), and it lets its own successor start only after that, so that what
// a successor reads ahead was complete when this stage began.
// Small stages are chains of barriers behind a launch, and the launch is what
// this hides: one client's whole step 303 -> 283 us, ExpandQuery of 32 clients
// 1.972 -> 1.956 ms.
__device__ __forceinline__ void let_next_stage_start() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void wait_for_previous_stage() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  let_next_stage_start();
}

// Thread-block cluster helpers: the CTAs of a tree node hand each other
// coefficient residues and partial sums through distributed shared memory.
// They are pushed: the receiver reads its own shared memory after the barrier,
// and no CTA has to outlive its peers' reads.
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Shared-memory address of the same offset in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t peer_addr(const void *local, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(local)), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_peer(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
// No memory ordering: for a CTA that is done reading its own shared memory.
__device__ __forceinline__ void cluster_arrive_relaxed() {
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

}  // namespace ntt

// Host side (ring_tables.cu): twiddle tables on the current device, built once
// per (device, N, primes) and kept for the process.
int ring_tables(const gpir_params_t *params, ntt::Ring *out);

}  // namespace gpir
