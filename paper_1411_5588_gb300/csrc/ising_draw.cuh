// Drawing and deciding a word of sites, split so that the random numbers need
// nothing of the lattice.
//
// A Metropolis decision compares a site's word u with a threshold that
// depends on the site's spin S and on k, its number of up neighbours.  Turning
// S round changes the sign of dE, so of the two moves at one k at most one
// costs energy: the other always happens.  One threshold t_k per k (k = 0 ..
// 6) therefore holds the whole table of a row class, and the bit mask
// M_k = [u < t_k] of a word's 32 sites can be drawn before the lattice is
// known: while the previous half-sweep is still running.  What is left once
// it has finished is bit logic on whole words:
//   flip = mux_k(M_k) | (S ^ mux_k(U_k)),
// U_k = all ones where the costly move at k starts from an up spin.
//
// Without a field on the layer (every inner layer when H = 0), M_k = M_{6-k}
// and k = 3 always flips: three masks.  The walls' layers and films in a bulk
// field take seven, which is half as long again.  Where a launch is bound by the
// integer pipes and not by its chain, those are drawn the other way round: once
// the lattice is known, a site's t_k is looked up in shared memory and its
// word compared with that one (draw_looked_up).
//
// Measured on GB300, register-only loops, cycles per 32-site word and warp
// scheduler: 16 products per Philox call alone 600; three masks 805; a table
// in shared memory, one look-up per site, 830.  So three masks cost no
// throughput, and move the draws out of the dependent chain.  120x240x1600 in a
// bulk field, per sweep: seven masks 63.1 us, look-ups 40.7 (without the field,
// three masks, 38.2).
#pragma once
#include <type_traits>

#include "ising_device.cuh"

namespace isg {

#ifdef __CUDACC__

template <int K>
struct Masks {
  uint32_t m[K];
};

// acc + BIT when u < t: each site's bit is set once, and unlike a predicated OR
// an add can go to either integer pipe.
template <uint32_t BIT>
__device__ __forceinline__ void put_if_lt(uint32_t& acc, uint32_t u, uint32_t t) {
  asm("{\n\t.reg .pred p;\n\tsetp.lt.u32 p, %1, %2;\n\t@p add.u32 %0, %0, %3;\n\t}"
      : "+r"(acc) : "r"(u), "r"(t), "n"(BIT));
}
__device__ __forceinline__ void put_if_lt_r(uint32_t& acc, uint32_t u, uint32_t t, uint32_t bit) {
  asm("{\n\t.reg .pred p;\n\tsetp.lt.u32 p, %1, %2;\n\t@p add.u32 %0, %0, %3;\n\t}"
      : "+r"(acc) : "r"(u), "r"(t), "r"(bit));
}

// The masks' bits of the four words u of one Philox call, bit Q + 8 i for word i.
template <uint32_t Q, int K>
__device__ __forceinline__ void put_call(Masks<K>& a, const uint32_t (&t)[K], const uint32_t (&u)[4]) {
#pragma unroll
  for (int k = 0; k < K; k++) {
    put_if_lt<1u << Q>(a.m[k], u[0], t[k]);
    put_if_lt<1u << (Q + 8)>(a.m[k], u[1], t[k]);
    put_if_lt<1u << (Q + 16)>(a.m[k], u[2], t[k]);
    put_if_lt<1u << (Q + 24)>(a.m[k], u[3], t[k]);
  }
}

template <int K>
__device__ __forceinline__ void masks_zero(Masks<K>& a) {
#pragma unroll
  for (int k = 0; k < K; k++) a.m[k] = 0;
}

// One word of R rows (bits j B + q + 8 i: row j's call q, B = 8 / R), R = 1: the
// eight calls from call number c1 on.  row, X: the first row and its parity
// array; ncalls: the calls of a row that hold sites (R = 1: of this word).
//
// Two calls are drawn side by side, two independent chains; where no word of
// the film has more than four calls (not paired: W = 1) each is drawn alone.
// The calls of a row are unrolled with immediate site bits; the rows of a packed
// word are a loop.  ROLL: a loop over the calls, one at a time.
template <int R, bool FULL, int K, bool ROLL = false>
__device__ __forceinline__ void draw_masks(Masks<K>& a, const uint32_t (&t)[K], uint32_t row, uint32_t X, uint32_t c1,
                                           uint32_t ncalls, bool paired, uint32_t sweep,
                                           const uint32_t* rk0, const uint32_t* rk1) {
  constexpr uint32_t B = 8 / R;
  masks_zero(a);
  if constexpr (ROLL) {
#pragma unroll 1
    for (uint32_t Q = 0; Q < 8; Q++) {
      const uint32_t q = R == 1 ? Q : Q % B, j = R == 1 ? 0u : Q / B;  // call q of row j
      if (q >= ncalls) continue;
      const PhiloxRow3 p(row + j, sweep, X ^ (j & 1u), rk0, rk1);
      uint32_t u[4];
      p.draw(c1 + q, u);
#pragma unroll
      for (int i = 0; i < 4; i++) {
#pragma unroll
        for (int k = 0; k < K; k++) put_if_lt_r(a.m[k], u[i], t[k], 1u << (Q + 8 * i));
      }
    }
    return;
  }
  // calls Q and Q + D side by side, from the word's call number c1 on
  auto two = [&](auto qc, auto dc, Masks<K>& s, const PhiloxRow3& p, bool second) {
    constexpr uint32_t Q = decltype(qc)::value, D = decltype(dc)::value;
    uint32_t u[4], v[4];
    p.draw2(c1 + Q, c1 + Q + D, u, v);
    put_call<Q>(s, t, u);
    if (second) put_call<Q + D>(s, t, v);
  };
  auto one = [&](auto qc, Masks<K>& s, const PhiloxRow3& p) {
    constexpr uint32_t Q = decltype(qc)::value;
    uint32_t u[4];
    p.draw(c1 + Q, u);
    put_call<Q>(s, t, u);
  };
  using I0 = std::integral_constant<uint32_t, 0>;
  using I1 = std::integral_constant<uint32_t, 1>;
  using I2 = std::integral_constant<uint32_t, 2>;
  using I3 = std::integral_constant<uint32_t, 3>;
  using I4 = std::integral_constant<uint32_t, 4>;
  if constexpr (R == 1) {
    const PhiloxRow3 p(row, sweep, X, rk0, rk1);
    if (FULL || paired || ncalls > 4) {
      two(I0{}, I4{}, a, p, FULL || ncalls > 4);
      if (FULL || ncalls > 1) two(I1{}, I4{}, a, p, FULL || ncalls > 5);
      if (FULL || ncalls > 2) two(I2{}, I4{}, a, p, FULL || ncalls > 6);
      if (FULL || ncalls > 3) two(I3{}, I4{}, a, p, FULL || ncalls > 7);
    } else {
      one(I0{}, a, p);
      if (ncalls > 1) one(I1{}, a, p);
      if (ncalls > 2) one(I2{}, a, p);
      if (ncalls > 3) one(I3{}, a, p);
    }
  } else {
#pragma unroll 1
    for (uint32_t j = 0; j < R; j++) {
      const PhiloxRow3 p(row + j, sweep, X ^ (j & 1u), rk0, rk1);
      Masks<K> s;
      masks_zero(s);
      if (ncalls > 1) two(I0{}, I1{}, s, p, true);
      else one(I0{}, s, p);
      if (R == 2 && ncalls > 3) two(I2{}, I1{}, s, p, true);
      else if (R == 2 && ncalls > 2) one(I2{}, s, p);
#pragma unroll
      for (int k = 0; k < K; k++) a.m[k] |= s.m[k] << (j * B);
    }
  }
}

__device__ __forceinline__ uint32_t maj3(uint32_t a, uint32_t b, uint32_t c) { return (a & b) | (c & (a ^ b)); }
__device__ __forceinline__ uint32_t mux(uint32_t c, uint32_t if1, uint32_t if0) { return (c & if1) | (~c & if0); }

// The words a decision needs, all on the sites of S: the x and y neighbours
// (wrap signs folded in, an empty slot 0) and the two z neighbours.
struct Hood {
  uint32_t S, xm, xp, ym, yp, z0, zs;
};

// k = c0 + 2 c1 + 4 c2, bit-sliced.
struct Count {
  uint32_t c0, c1, c2;
};

__device__ __forceinline__ Count count_up(const Hood& h) {
  const uint32_t s1 = h.xm ^ h.xp ^ h.ym, k1 = maj3(h.xm, h.xp, h.ym);
  const uint32_t s2 = h.yp ^ h.z0 ^ h.zs, k2 = maj3(h.yp, h.z0, h.zs);
  const uint32_t k3 = s1 & s2;
  return Count{s1 ^ s2, k1 ^ k2 ^ k3, maj3(k1, k2, k3)};
}

// Sites that flip, three masks m = {M_4 = M_2, M_5 = M_1, M_6 = M_0}.
__device__ __forceinline__ uint32_t flips3(uint32_t S, const Count& c, uint32_t m4, uint32_t m5, uint32_t m6) {
  const uint32_t even = mux(c.c1 ^ c.c2, m4, m6);  // k = 2, 4: m4; 0, 6: m6
  const uint32_t odd = m5 | c.c1;                  // k = 1, 5: m5; 3: always
  return mux(c.c0, odd, even) | (S ^ c.c2);
}

// The general form; up, frz: ClassDraw's bits.
__device__ __forceinline__ uint32_t mux7(const Count& c, const uint32_t (&v)[7]) {
  const uint32_t e0 = mux(c.c0, v[1], v[0]), e1 = mux(c.c0, v[3], v[2]), e2 = mux(c.c0, v[5], v[4]);
  return mux(c.c2, mux(c.c1, v[6], e2), mux(c.c1, e1, e0));
}
__device__ __forceinline__ uint32_t bits7(const Count& c, uint32_t bits) {
  uint32_t v[7];
#pragma unroll
  for (int k = 0; k < 7; k++) v[k] = (bits >> k) & 1u ? 0xFFFFFFFFu : 0u;
  return mux7(c, v);
}
__device__ __forceinline__ uint32_t flips7(uint32_t S, const Count& c, const uint32_t (&m)[7], uint32_t up,
                                           uint32_t frz) {
  uint32_t fl = mux7(c, m) | (S ^ bits7(c, up));
  if (frz) fl &= ~bits7(c, frz);
  return fl;
}

// Thresholds of the four row classes for look-ups by k, t[k] of class c at 8 c + k:
// 32 words in as many banks of shared memory, so that no two sites conflict.
constexpr uint32_t kLookWords = 32;

// The thresholds of the four sites of one call: byte i of `at` is site i's byte
// offset in the table.
__device__ __forceinline__ void look_up(uint32_t (&t)[4], const uint32_t* look, uint32_t at) {
#pragma unroll
  for (uint32_t i = 0; i < 4; i++)
    t[i] = *reinterpret_cast<const uint32_t*>(reinterpret_cast<const char*>(look) + __byte_perm(at, 0u, 0x4440u + i));
}

// The mask [u < t_k] of a word whose counts k are known, class cl: one comparison
// per site with a looked-up threshold, where the general form compares each site
// with all seven.  The arguments are draw_masks'.  HOW (R = 1): eight calls in
// straight-line code, so that one pair's look-ups pass under another's draws; the
// same with only the word's calls, in branches; or those as a loop, in fewer
// registers.
enum : int { kLookLoop, kLookBranches, kLookStraight };
template <int R, int HOW>
__device__ __forceinline__ uint32_t draw_looked_up(const Count& k, const uint32_t* look, uint32_t cl, uint32_t row,
                                                   uint32_t X, uint32_t c1, uint32_t ncalls, uint32_t sweep,
                                                   const uint32_t* rk0, const uint32_t* rk1) {
  const uint32_t base = cl * 0x20202020u;  // the class's part of the offsets
  uint32_t acc = 0;
  uint32_t u[4], v[4], tu[4], tv[4];
  auto put = [](uint32_t& s, auto at, const uint32_t (&x)[4], const uint32_t (&t)[4]) {
    constexpr uint32_t A = decltype(at)::value;
    put_if_lt<1u << A>(s, x[0], t[0]);
    put_if_lt<1u << (A + 8)>(s, x[1], t[1]);
    put_if_lt<1u << (A + 16)>(s, x[2], t[2]);
    put_if_lt<1u << (A + 24)>(s, x[3], t[3]);
  };
  using I0 = std::integral_constant<uint32_t, 0>;
  using I1 = std::integral_constant<uint32_t, 1>;
  using I2 = std::integral_constant<uint32_t, 2>;
  using I3 = std::integral_constant<uint32_t, 3>;
  using I4 = std::integral_constant<uint32_t, 4>;
  // y[q]: the counts of the sites at bits q and q + 4 of each byte, in its low and
  // its high nibble
  const uint32_t p0 = (k.c0 & 0x55555555u) | ((k.c1 << 1) & 0xAAAAAAAAu);
  const uint32_t p1 = ((k.c0 >> 1) & 0x55555555u) | (k.c1 & 0xAAAAAAAAu);
  const uint32_t y0 = (p0 & 0x33333333u) | ((k.c2 << 2) & 0x44444444u);
  const uint32_t y1 = (p1 & 0x33333333u) | ((k.c2 << 1) & 0x44444444u);
  const uint32_t y2 = ((p0 >> 2) & 0x33333333u) | (k.c2 & 0x44444444u);
  const uint32_t y3 = ((p1 >> 2) & 0x33333333u) | ((k.c2 >> 1) & 0x44444444u);
  if constexpr (R == 1 && HOW == kLookStraight) {
    // calls q and q + 4 side by side
    const PhiloxRow3 p(row, sweep, X, rk0, rk1);
    auto two = [&](auto qc, uint32_t y) {
      constexpr uint32_t q = decltype(qc)::value;
      look_up(tu, look, ((y << 2) & 0x3C3C3C3Cu) | base);
      look_up(tv, look, ((y >> 2) & 0x3C3C3C3Cu) | base);
      p.draw2(c1 + q, c1 + q + 4, u, v);
      put(acc, qc, u, tu);
      put(acc, std::integral_constant<uint32_t, q + 4>{}, v, tv);
    };
    two(I0{}, y0);
    two(I1{}, y1);
    two(I2{}, y2);
    two(I3{}, y3);
  } else if constexpr (R == 1) {
    // the same, for a row's only word with fewer than eight calls
    const PhiloxRow3 p(row, sweep, X, rk0, rk1);
    auto some = [&](uint32_t q) {
      if (q >= ncalls) return;
      const uint32_t y = q == 0 ? y0 : q == 1 ? y1 : q == 2 ? y2 : y3;
      uint32_t s = 0;
      look_up(tu, look, ((y << 2) & 0x3C3C3C3Cu) | base);
      if (q + 4 < ncalls) {
        look_up(tv, look, ((y >> 2) & 0x3C3C3C3Cu) | base);
        p.draw2(c1 + q, c1 + q + 4, u, v);
        put(s, I4{}, v, tv);
      } else {
        p.draw(c1 + q, u);
      }
      put(s, I0{}, u, tu);
      acc |= s << q;
    };
    if constexpr (HOW == kLookBranches) {
      some(0);
      some(1);
      some(2);
      some(3);
    } else {
#pragma unroll 1
      for (uint32_t q = 0; q < 4; q++) some(q);
    }
  } else {
    // row j's calls q and q + 1 side by side: bits b and b + 1 of a byte
    constexpr uint32_t B = 8 / R;
#pragma unroll 1
    for (uint32_t b = 0; b < 8; b += 2) {
      const uint32_t j = b / B, q = b % B;
      if (q >= ncalls) continue;
      const uint32_t ya = ((b & 2u) ? y2 : y0) >> (b & 4u), yb = ((b & 2u) ? y3 : y1) >> (b & 4u);
      const PhiloxRow3 p(row + j, sweep, X ^ (j & 1u), rk0, rk1);
      uint32_t s = 0;
      look_up(tu, look, ((ya << 2) & 0x3C3C3C3Cu) | base);
      if (q + 1 < ncalls) {
        look_up(tv, look, ((yb << 2) & 0x3C3C3C3Cu) | base);
        p.draw2(c1 + q, c1 + q + 1, u, v);
        put(s, I1{}, v, tv);
      } else {
        p.draw(c1 + q, u);
      }
      put(s, I0{}, u, tu);
      acc |= s << b;
    }
  }
  return acc;
}

// Sites that flip, mask m = [u < t_k].
__device__ __forceinline__ uint32_t flips_looked_up(uint32_t S, const Count& c, uint32_t m, const ClassDraw& cl) {
  // the usual orders of k: with a small field, or none, the costly move starts
  // from an up spin for k >= 4 or k >= 3
  const uint32_t up = cl.up == 0x70u ? c.c2 : cl.up == 0x78u ? c.c2 | (c.c0 & c.c1) : bits7(c, cl.up);
  uint32_t fl = m | (S ^ up);
  if (cl.alw) fl |= bits7(c, cl.alw);
  if (cl.frz) fl &= ~bits7(c, cl.frz);
  return fl;
}

// sum over the valid sites of s (2 k - D): the bonds from the word's sites
// (new value v) to their neighbours, D bond slots each.
__device__ __forceinline__ int word_bond_sum(const Count& c, uint32_t v, uint32_t valid, int D) {
  const int kv = __popc(c.c0 & v) + 2 * __popc(c.c1 & v) + 4 * __popc(c.c2 & v);
  const int ka = __popc(c.c0 & valid) + 2 * __popc(c.c1 & valid) + 4 * __popc(c.c2 & valid);
  return 4 * kv - 2 * ka - D * (2 * __popc(v) - __popc(valid));
}

// z neighbours of a word of R packed rows: site l - 1 of each row for prev,
// l + 1 for next, the rows' ends joined (first: the rows' first-site bits;
// pos: the bit of their last site relative to those; top: the last call's
// bits of each row).  Padding bits of v are 0.
__device__ __forceinline__ uint32_t packed_prev(uint32_t v, uint32_t first, uint32_t pos) {
  return (v << 8) | ((v >> 23) & 0xFEu & ~first) | ((v >> pos) & first);
}
__device__ __forceinline__ uint32_t packed_next(uint32_t v, uint32_t first, uint32_t pos) {
  // byte 0 shifted down by one call, its rows' first sites left out (they are
  // the row before's in the packed word), lands in byte 3
  return (v >> 8) | (((v & ~first) << 23) & 0x7F000000u) | ((v & first) << pos);
}

#endif  // __CUDACC__

}  // namespace isg
