// CUDA kernels of the Ising-film sweep for sm_103a.
//
//  - update_kernel, update_film_kernel: one half-sweep (colour c) of every film
//    of a launch, of one film.  The four phases of a sweep (Appendix
//    checkerboard, split by the Eq. 11 wrap rows) run as two launches: the
//    thread that decides a word of row (kx, 1) decides the word of row (kx', Ly)
//    whose wrap neighbour it is right after it -- kx' = Lx+1-kx for the Eq. 11
//    rule, kx' = kx otherwise.  That row depends on nothing else updated in the
//    half-sweep, so the thread-local order reproduces "all of {c, ky<Ly}, then
//    all of {c, ky=Ly}" exactly.  The half-sweep 1 launch of a sweep after which
//    films record also sums their int64 record quantities B, M, M1, Mn and
//    m(kx) (Eqs. 1, 7, 9, 17, 19) from the words it holds in registers, into
//    per-layer accumulators.
//  - slab_kernel: every sweep of a call with the film in shared memory, of one
//    CTA (the resident path) or of a cluster's CTAs.
//  Where a half-sweep is bound by its chain, a word's random numbers are drawn
//  and compared before its lattice neighbourhood is known (ising_draw.cuh), so
//  the wait for the previous half-sweep -- a launch or a barrier -- hides behind
//  the draws.
//  - record_kernel: writes those records and clears the accumulators.
//  - measure_partial_kernel / measure_finalize_kernel: the same sums from the
//    lattice alone (an on-demand measurement), per-block partials in a
//    scratch area, then one block per film writes the record.
//  - init_kernel, pack_kernel, unpack_kernel, advance_kernel.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "ising_draw.cuh"

#include "ising_launch.h"

namespace isg {

namespace cg = cooperative_groups;

namespace {

// Programmatic dependent launch: every kernel of the sweep path lets the next
// launch of its stream start early (its blocks then sit in pdl_wait) and
// waits, before it touches any film state, for the previous grid to complete
// and its writes to be visible.  Without the launch attribute both are no-ops.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Checked builds (-DISING_CHECKED) test every lattice word index against its
// plane before the access: an index out of range is counted, the first one
// is kept (site << 48 | index), and the access goes to word 0 instead (a
// store is dropped).  Normal builds compile the checks away.
#ifdef ISING_CHECKED
__device__ unsigned long long g_oob_count;
__device__ unsigned long long g_oob_first;
__device__ __forceinline__ bool oob(uint64_t idx, uint64_t lim, uint32_t site) {
  if (idx < lim) return false;
  atomicAdd(&g_oob_count, 1ull);
  atomicCAS(&g_oob_first, 0ull, ((unsigned long long)site << 48) | (idx & 0xFFFFFFFFFFFFull));
  return true;
}
#define ISG_LD(p, idx, lim, site) ((p)[oob((idx), (lim), (site)) ? 0 : (idx)])
#define ISG_ST(p, idx, lim, site, v) \
  do {                               \
    if (!oob((idx), (lim), (site))) (p)[(idx)] = (v); \
  } while (0)
#else
#define ISG_LD(p, idx, lim, site) ((void)(lim), (p)[(idx)])
#define ISG_ST(p, idx, lim, site, v) ((void)(lim), (p)[(idx)] = (v))
#endif

__host__ __device__ inline uint32_t seam_joins_one_colour(uint32_t Lx, uint32_t Ly, uint32_t y_mode) {
  return y_mode == kYGapbc ? ((Lx + Ly) % 2 == 0) : (Ly % 2 == 1);
}

// Whether film F, at chunk start sweep `sweep`, records after `done` sweeps
// of the chunk.
__device__ __forceinline__ bool records_after(const FilmDesc& F, uint32_t sweep, uint32_t done) {
  if (F.measure_every == 0 || done == 0 || F.sweep_end - sweep < done) return false;
  return ((sweep + done) % F.measure_every) == 0;
}

__device__ __forceinline__ bool measured_now(const FilmDesc& F, uint32_t done, int force) {
  return force || records_after(F, F.sweep, done);
}

__device__ __forceinline__ int64_t block_sum(int64_t v, int64_t* s_red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xFFFFFFFFu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) s_red[warp] = v;
  __syncthreads();
  int64_t t = 0;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x >> 5); i++) t += s_red[i];
  __syncthreads();
  return t;  // valid in thread 0
}

// The record of film Fg after `done` sweeps of the chunk (chunk-start sweep
// `sweep`), from the per-layer accumulators half-sweep 1 filled, which it
// clears; advances the film's ring counter.  F holds the film's static
// fields (a staged copy or Fg itself).  The whole block calls it; s_red holds
// one int64 per warp.
__device__ __noinline__ void write_record(FilmDesc* Fg, const FilmDesc& F, uint32_t sweep, int64_t* part,
                                             int64_t* records, uint32_t done, int64_t* s_red, uint32_t* s_slot) {
  const uint32_t Lx = F.Lx;
  uint32_t rn = 0;
  __syncthreads();
  if (threadIdx.x == 0) {
    rn = __ldcg(&Fg->rec_next);  // written by an earlier kernel
    *s_slot = F.rec_cap ? rn % F.rec_cap : 0u;
  }
  __syncthreads();
  int64_t* rec = records + F.rec_off + (size_t)*s_slot * (5 + Lx);
  int64_t* acc = part + acc_offset(F);
  int64_t M = 0, Bs = 0;
  for (uint32_t kx = threadIdx.x; kx < Lx; kx += blockDim.x) {
    const int64_t m = acc[2 * kx], b = acc[2 * kx + 1];
    acc[2 * kx] = 0;
    acc[2 * kx + 1] = 0;
    rec[5 + kx] = m;
    M += m;
    Bs += b;
  }
  const int64_t tM = block_sum(M, s_red);
  const int64_t tB = block_sum(Bs, s_red);
  if (threadIdx.x == 0) {
    rec[0] = (int64_t)sweep + done;
    rec[1] = tB;
    rec[2] = tM;
    rec[3] = rec[5];
    rec[4] = rec[5 + Lx - 1];
    Fg->rec_next = rn + 1;
  }
}

// One word's record sums; layer: 0-based kx, none when 0xFFFFFFFF.
struct LayerSums {
  uint32_t layer = 0xFFFFFFFFu;
  int m = 0, b = 0;
};

// Adds the sums of every lane that has some into the film's per-layer int64
// accumulators [2 kx (magnetisation), 2 kx + 1 (bonds)].  All 32 lanes call
// it.  The lanes in the first active lane's layer add with two warp
// reductions and two atomics; any other lane adds its own.  Integer atomics
// are exact in any order.
__device__ __forceinline__ void add_layer_sums(unsigned long long* acc, const LayerSums& r) {
  const bool on = r.layer != 0xFFFFFFFFu;
  const uint32_t act = __ballot_sync(0xFFFFFFFFu, on);
  if (act == 0) return;
  const int lead = __ffs(act) - 1;
  const uint32_t l0 = __shfl_sync(0xFFFFFFFFu, r.layer, lead);
  const bool in0 = on && r.layer == l0;
  const int m = __reduce_add_sync(0xFFFFFFFFu, in0 ? r.m : 0);
  const int b = __reduce_add_sync(0xFFFFFFFFu, in0 ? r.b : 0);
  if ((int)(threadIdx.x & 31u) == lead) {
    atomicAdd(acc + 2 * (size_t)l0, (unsigned long long)(long long)m);
    atomicAdd(acc + 2 * (size_t)l0 + 1, (unsigned long long)(long long)b);
  } else if (on && !in0) {
    atomicAdd(acc + 2 * (size_t)r.layer, (unsigned long long)(long long)r.m);
    atomicAdd(acc + 2 * (size_t)r.layer + 1, (unsigned long long)(long long)r.b);
  }
}

// A lane's own sums, without a warp reduction (partner words: a few lanes).
__device__ __forceinline__ void add_lane_sums(unsigned long long* acc, const LayerSums& r) {
  if (r.layer == 0xFFFFFFFFu) return;
  atomicAdd(acc + 2 * (size_t)r.layer, (unsigned long long)(long long)r.m);
  atomicAdd(acc + 2 * (size_t)r.layer + 1, (unsigned long long)(long long)r.b);
}


// ------------------------------------------------------------ grid path

// Per-launch constants of one film.
struct FilmCtx {
  uint32_t* plane0;
  uint32_t* plane1;
  uint32_t Lx, Ly, W, y_mode, x_pbc, last_mask, last_calls;
  uint32_t pos;          // bit of a row's last site in its last word
  uint32_t plane_words;  // words of one plane (Lx * Ly * W), for checked builds
  uint32_t neg;          // all ones where the y wrap reverses the sign
  uint32_t seam_same;    // the y-wrap bonds join sites of one colour (Lx+Ly even under Eq. 11, Ly odd otherwise)
  const ClassDraw* cls;
  const uint32_t* rk0;   // Philox round keys (constant bank or shared memory)
  const uint32_t* rk1;
  uint32_t colour, sweep;
};

__device__ __forceinline__ void film_ctx(FilmCtx& c, const FilmDesc& d, uint32_t* pool, uint32_t colour,
                                         uint32_t sweep) {
  c.Lx = d.Lx; c.Ly = d.Ly; c.W = d.W;
  c.y_mode = d.y_mode; c.x_pbc = d.x_pbc;
  c.last_mask = d.last_mask; c.last_calls = d.last_calls;
  c.pos = bitpos((d.n - 1) & 31u);
  c.plane_words = d.Lx * d.Ly * d.W;
  c.neg = d.y_mode != kYPbc ? 0xFFFFFFFFu : 0u;
  c.seam_same = seam_joins_one_colour(d.Lx, d.Ly, d.y_mode);
  c.cls = d.cls; c.rk0 = d.rk0; c.rk1 = d.rk1;
  c.colour = colour; c.sweep = sweep;
  c.plane0 = pool + d.spin_off;
  c.plane1 = c.plane0 + (size_t)d.Lx * d.Ly * d.W;
}

// Fills the block's threshold table for look-ups (the caller synchronises).
__device__ __forceinline__ void fill_look(uint32_t* look, const ClassDraw* cls) {
  if (threadIdx.x < kLookWords) {
    const uint32_t k = threadIdx.x & 7u;
    look[threadIdx.x] = k < 7 ? cls[threadIdx.x >> 3].t[k] : 0u;
  }
}

// The masks of a word drawn ahead: the three-mask form fills m[4..6].
struct Drawn {
  uint32_t m[7];
};

// Masks of one word of R rows from row `row` (parity array X) of class cl;
// any7: the warp takes the general form (ROLL: as a loop over the calls, in
// fewer registers: the general form of one word per thread then keeps to the 64
// of eight blocks per SM).  calls: the word's (R > 1: a row's) Philox calls;
// full: every word of the film has eight.
template <int R, bool ROLL = false>
__device__ __forceinline__ void draw_any(Drawn& o, bool any7, const ClassDraw& cl, uint32_t row, uint32_t X,
                                         uint32_t w, uint32_t calls, bool full, bool paired, uint32_t sweep,
                                         const uint32_t* rk0, const uint32_t* rk1) {
  if (!any7) {
    Masks<3> a;
    const uint32_t t[3] = {cl.t[4], cl.t[5], cl.t[6]};
    if (R == 1 && full) draw_masks<1, true, 3>(a, t, row, X, 8u * w, 8u, true, sweep, rk0, rk1);
    else draw_masks<R, false, 3>(a, t, row, X, 8u * w, calls, paired, sweep, rk0, rk1);
    // all ones where t_k would be 2^32 (T = infinity)
    if (cl.alw & 0x70u) {
#pragma unroll
      for (int k = 0; k < 3; k++)
        if ((cl.alw >> (4 + k)) & 1u) a.m[k] = 0xFFFFFFFFu;
    }
    // every mask is set, so that none is live from one drawing to the next
    o = Drawn{{0, 0, 0, 0, a.m[0], a.m[1], a.m[2]}};
  } else {
    Masks<7> a;
    draw_masks<R, false, 7, ROLL>(a, cl.t, row, X, 8u * w, calls, paired, sweep, rk0, rk1);
#pragma unroll
    for (int k = 0; k < 7; k++) o.m[k] = (cl.alw >> k) & 1u ? 0xFFFFFFFFu : a.m[k];
  }
}

// The sites of a word that flip, by look-ups.  Words of rows of several take the
// straight-line form for eight calls, the partial last ones too (their warps
// have full ones, and what is drawn beyond the row's end is not valid).  So do
// rows of one partial word, in the grid kernels from five calls up (64 films of
// 64x128x48, six calls: 28.4 us per sweep, 30.4 as a loop), on slabs from seven (300
// films of 24x60x40, five calls, on a CTA each: 24.4 us in branches, 27.6 straight
// and as a loop).
template <int R, bool SLAB = false>
__device__ __forceinline__ uint32_t look_and_decide(const Hood& h, const Count& k, const uint32_t* look, uint32_t ci,
                                                    const ClassDraw& cl, uint32_t row, uint32_t X, uint32_t w,
                                                    uint32_t calls, bool several, uint32_t sweep,
                                                    const uint32_t* rk0, const uint32_t* rk1) {
  uint32_t m;
  if (R == 1 && (several || calls >= (SLAB ? 7u : 5u)))
    m = draw_looked_up<R, kLookStraight>(k, look, ci, row, X, 8u * w, 8u, sweep, rk0, rk1);
  else
    m = draw_looked_up<R, SLAB ? kLookBranches : kLookLoop>(k, look, ci, row, X, 8u * w, calls, sweep, rk0, rk1);
  return flips_looked_up(h.S, k, m, cl);
}

__device__ __forceinline__ uint32_t decide(const Hood& h, const Count& k, bool any7, const Drawn& a,
                                           const ClassDraw& cl) {
  if (!any7) return flips3(h.S, k, a.m[4], a.m[5], a.m[6]);
  return flips7(h.S, k, a.m, cl.up, cl.frz);
}

// Slot masks of a word of R packed rows: the rows' first-site bits, and the
// bits of row 0.
template <int R>
__device__ __forceinline__ constexpr uint32_t first_bits() {
  return R == 1 ? 0x01u : R == 2 ? 0x11u : 0x55u;
}
template <int R>
__device__ __forceinline__ constexpr uint32_t slot_mask() {
  return 0x01010101u * ((1u << (8 / R)) - 1u);
}

// The words of word w of row (kx, ky).
__device__ __forceinline__ void fetch_row(const FilmCtx& c, uint32_t kx, uint32_t ky, uint32_t w, Hood& f) {
  const uint32_t Lx = c.Lx, Ly = c.Ly, W = c.W;
  const uint32_t row = (kx - 1) * Ly + (ky - 1);
  const uint32_t X = (kx + ky + 1 + c.colour) & 1u;
  const uint32_t* __restrict__ P = X ? c.plane1 : c.plane0;
  const uint32_t* __restrict__ Q = X ? c.plane0 : c.plane1;
  const uint32_t rbase = row * W;  // planes hold < 2^31 words
  const uint32_t base = rbase + w;
  const uint32_t LyW = Ly * W;
  const uint32_t gkx = (c.y_mode == kYGapbc) ? (Lx - kx) : (kx - 1);  // 0-based layer of the wrap row
  const uint32_t lim = c.plane_words;
  f.S = ISG_LD(P, base, lim, 1);
  f.xm = (kx > 1) ? ISG_LD(P, base - LyW, lim, 2)
                  : (c.x_pbc ? ISG_LD(P, base + (Lx - 1) * LyW, lim, 3) : 0u);
  f.xp = (kx < Lx) ? ISG_LD(P, base + LyW, lim, 4)
                   : (c.x_pbc ? ISG_LD(P, base - (Lx - 1) * LyW, lim, 5) : 0u);
  f.ym = (ky > 1) ? ISG_LD(P, base - W, lim, 6) : (ISG_LD(P, (gkx * Ly + (Ly - 1)) * W + w, lim, 7) ^ c.neg);
  f.yp = (ky < Ly) ? ISG_LD(P, base + W, lim, 8) : (ISG_LD(P, gkx * LyW + w, lim, 9) ^ c.neg);
  f.z0 = ISG_LD(Q, base, lim, 10);
  // the second z neighbour: site j of array 0 meets site j - 1 of array 1,
  // site j of array 1 meets site j + 1 of array 0, the row's ends joined
  if (W == 1) {
    f.zs = X ? packed_next(f.z0, 1u, c.pos) : packed_prev(f.z0, 1u, c.pos);
  } else if (X == 0) {
    const uint32_t pw = (w > 0) ? ISG_LD(Q, base - 1, lim, 11) >> 31 : (ISG_LD(Q, rbase + W - 1, lim, 12) >> c.pos) & 1u;
    f.zs = shift_prev(f.z0, pw << 31);
  } else {
    const bool last = w + 1 == W;
    const uint32_t nw = last ? ISG_LD(Q, rbase, lim, 14) : ISG_LD(Q, base + 1, lim, 13);
    f.zs = shift_next(f.z0, 0u) | ((nw & 1u) << (last ? c.pos : 31u));
  }
}

// The same for R rows (kx, ky .. ky+R-1) of one-word rows, packed.
//
// Thin films: a film whose rows hold one partial word per parity array
// (W = 1) with at most 8 sites (R = 4) or 16 sites (R = 2) per array would
// spend the per-word work on a quarter or a half of a word's 32 sites.  Row
// j's bits, which sit in the low B = 8/R bits of each byte, move up by j*B
// bits into one register: packed bit j*B + q + 8*i is row j's site 4q + i,
// served by that row's Philox call q.  Consecutive rows update opposite
// arrays, and none reads an array another updates in the same half-sweep.
template <int R>
__device__ __forceinline__ void fetch_rows(const FilmCtx& c, uint32_t kx, uint32_t ky, uint32_t w, Hood& p) {
  if constexpr (R == 1) {
    fetch_row(c, kx, ky, w, p);
  } else {
    constexpr uint32_t B = 8 / R;
    p = Hood{0, 0, 0, 0, 0, 0, 0};
#pragma unroll
    for (uint32_t j = 0; j < R; j++) {
      Hood f;
      fetch_row(c, kx, ky + j, 0, f);
      const uint32_t sh = j * B, valid = c.last_mask;
      p.S |= f.S << sh;
      p.xm |= f.xm << sh;
      p.xp |= f.xp << sh;
      p.ym |= (f.ym & valid) << sh;
      p.yp |= (f.yp & valid) << sh;
      p.z0 |= f.z0 << sh;
      p.zs |= (f.zs & valid) << sh;
    }
  }
}

template <int R>
__device__ __forceinline__ void store_rows(const FilmCtx& c, uint32_t kx, uint32_t ky, uint32_t w, uint32_t v) {
#pragma unroll
  for (uint32_t j = 0; j < R; j++) {
    const uint32_t row = (kx - 1) * c.Ly + (ky + j - 1);
    const uint32_t X = (kx + ky + j + 1 + c.colour) & 1u;
    uint32_t* __restrict__ P = X ? c.plane1 : c.plane0;
    ISG_ST(P, row * c.W + w, c.plane_words, 16, R == 1 ? v : (v >> (j * (8 / R))) & slot_mask<R>());
  }
}

// A word of array X at an offset from a word of it, for columns.
__device__ __forceinline__ uint32_t col_ld(const FilmCtx& c, const uint32_t* p, ptrdiff_t off, uint32_t X,
                                           uint32_t site) {
#ifdef ISING_CHECKED
  const uint32_t* base = X ? c.plane1 : c.plane0;
  return ISG_LD(base, (uint64_t)(p + off - base), c.plane_words, site);
#else
  return p[off];
#endif
}
__device__ __forceinline__ void col_st(const FilmCtx& c, const uint32_t* p, uint32_t X, uint32_t v) {
  uint32_t* base = X ? c.plane1 : c.plane0;
#ifdef ISING_CHECKED
  ISG_ST(base, (uint64_t)(p - base), c.plane_words, 16, v);
#else
  (void)base;
  *const_cast<uint32_t*>(p) = v;
#endif
}

// Bond slots of a site of layer kx.
__device__ __forceinline__ int bond_slots(uint32_t kx, uint32_t Lx, uint32_t x_pbc) {
  return 4 + ((kx > 1 || x_pbc) ? 1 : 0) + ((kx < Lx || x_pbc) ? 1 : 0);
}

// Record sums of half-sweep 1.  Every neighbour word a thread loaded is final
// after it -- it holds the other colour -- except the -y word of a ky = 1 row
// when the seam joins one colour: that is its wrap partner, which the same
// thread updates right after it.  So each thread adds up, for its word, the
// magnetisation of the row's two words and sum sigma_b S_i S_j over the bonds
// from the word's sites to their neighbours (an empty x slot is no bond), and
// every bond of the film is counted once.
__device__ __forceinline__ LayerSums word_sums(uint32_t kx, const Count& k, uint32_t v, uint32_t z0, uint32_t valid,
                                               int D) {
  LayerSums r;
  r.layer = kx - 1;
  r.b = word_bond_sum(k, v, valid, D);
  r.m = 2 * (__popc(v) + __popc(z0)) - 2 * __popc(valid);
  return r;
}

// Seam correction of a ky = 1 word (new value v, other word z0) and its
// partner word (old value S2, other word z2; the partner row is its slot at
// bit shift sh) when the seam joins one colour: the first word's -y count used
// the partner's old word, so it comes out again (the partner counts that bond
// from its +y side with both final words), and the seam bonds between the two
// rows' other arrays, which no one else holds, go in.
__device__ __forceinline__ int seam_adjust(uint32_t v, uint32_t z0, uint32_t S2, uint32_t z2, uint32_t sh,
                                           uint32_t neg, uint32_t valid) {
  const int nv = __popc(valid);
  const int stale = 2 * __popc(~(v ^ (S2 >> sh) ^ neg) & valid) - nv;
  const int other = nv - 2 * __popc((z0 ^ (z2 >> sh)) & valid);
  return (neg ? -other : other) - stale;
}

// The word of group (kx, ky) and, for a pair, its wrap partner's after it, by
// look-ups, once the previous launch is complete: nothing is drawn ahead, but a
// general word is drawn in two thirds of the masks' time.
template <int R, bool MEAS>
__device__ __forceinline__ void update_looked_up(const FilmCtx& c, const uint32_t* look, uint32_t kx, uint32_t ky,
                                                 uint32_t w, bool pair, uint32_t calls, uint32_t valid, uint32_t valid1,
                                                 bool meas, LayerSums& r1, LayerSums& r2) {
  constexpr uint32_t B = 8 / R, kSeam = (R - 1) * B;  // the partner row's slot: the last of its group
  const uint32_t kx2 = (c.y_mode == kYGapbc) ? c.Lx + 1 - kx : kx, ky2 = c.Ly - R + 1;
  Hood h, g;
  fetch_rows<R>(c, kx, ky, w, h);
  if (pair) fetch_rows<R>(c, kx2, ky2, w, g);
  uint32_t v1 = 0, z1 = 0;
#pragma unroll 1
  for (uint32_t r = 0; r < (pair ? 2u : 1u); r++) {
    const uint32_t x = r ? kx2 : kx, y = r ? ky2 : ky, cl = row_class(x, c.Lx);
    if (r) {
      // the partner's wrap neighbour is the word just decided where the seam
      // joins one colour
      if (c.seam_same) g.yp = (g.yp & ~(valid1 << kSeam)) | (((v1 ^ c.neg) & valid1) << kSeam);
      h = g;
    }
    const Count k = count_up(h);
    const uint32_t v =
        h.S ^ (look_and_decide<R>(h, k, look, cl, c.cls[cl], (x - 1) * c.Ly + y - 1, (x + y + 1 + c.colour) & 1u, w,
                                            calls, c.W > 1, c.sweep, c.rk0, c.rk1) & valid);
    store_rows<R>(c, x, y, w, v);
    if (MEAS && meas) {
      LayerSums q = word_sums(x, k, v, h.z0, valid, bond_slots(x, c.Lx, c.x_pbc));
      if (r && c.seam_same) q.b += seam_adjust(v1, z1, h.S, h.z0, kSeam, c.neg, valid1);
      if (r) r2 = q;
      else r1 = q;
    }
    v1 = v;
    z1 = h.z0;
  }
}

// The pair of a ky = 1 word (group 0 of layer kx) and its wrap partner's, row Ly
// of layer kx' (= Lx + 1 - kx under Eq. 11, else kx), in this order.
template <int R, bool MEAS, class Wait, class AccOf>
__device__ __forceinline__ void update_pair(const FilmCtx& c, uint32_t kx, uint32_t w, uint32_t calls, uint32_t valid,
                                            uint32_t valid1, bool meas, AccOf acc_of, Wait wait) {
  constexpr uint32_t B = 8 / R, kSeam = (R - 1) * B;  // the partner row's slot: the last of its group
  const uint32_t kx2 = (c.y_mode == kYGapbc) ? c.Lx + 1 - kx : kx, ky2 = c.Ly - R + 1;
  const uint32_t c1 = row_class(kx, c.Lx), c2 = row_class(kx2, c.Lx);
  const bool any7 = !c.cls[c1].sym || !c.cls[c2].sym;
  Drawn a[2];
#pragma unroll 1
  for (uint32_t n = 0; n < 2; n++) {
    const uint32_t k = n ? kx2 : kx, ky = n ? ky2 : 1u;
    Drawn x;
    draw_any<R, true>(x, any7, c.cls[n ? c2 : c1], (k - 1) * c.Ly + ky - 1, (k + ky + 1 + c.colour) & 1u, w, calls,
                      c.last_mask == 0xFFFFFFFFu, c.W > 1, c.sweep, c.rk0, c.rk1);
    if (n == 0) a[0] = x;
    else a[1] = x;
  }
  wait();
  Hood h, g;
  fetch_rows<R>(c, kx, 1, w, h);
  fetch_rows<R>(c, kx2, ky2, w, g);
  const Count k = count_up(h);
  const uint32_t v = h.S ^ (decide(h, k, any7, a[0], c.cls[c1]) & valid);
  store_rows<R>(c, kx, 1, w, v);
  // the partner's wrap neighbour is the word just decided where the seam joins
  // one colour
  if (c.seam_same) g.yp = (g.yp & ~(valid1 << kSeam)) | (((v ^ c.neg) & valid1) << kSeam);
  const Count k2 = count_up(g);
  const uint32_t v2 = g.S ^ (decide(g, k2, any7, a[1], c.cls[c2]) & valid);
  store_rows<R>(c, kx2, ky2, w, v2);
  if (MEAS && meas) {
    add_lane_sums(acc_of(), word_sums(kx, k, v, h.z0, valid, bond_slots(kx, c.Lx, c.x_pbc)));
    LayerSums q = word_sums(kx2, k2, v2, g.z0, valid, bond_slots(kx2, c.Lx, c.x_pbc));
    if (c.seam_same) q.b += seam_adjust(v, h.z0, g.S, g.z0, kSeam, c.neg, valid1);
    add_lane_sums(acc_of(), q);
  }
}

// Column rp - Lx (behind the pairs) of shape `items`: groups g .. g1 - 1 of layer
// kx; the two walls' columns come first (grid_columns).
struct GridColumn {
  bool on;
  uint32_t kx, g, g1;
};
template <int R>
__device__ __forceinline__ GridColumn grid_column(const FilmDesc& d, uint32_t items, uint32_t rp) {
  const uint32_t rq = rp < d.Lx ? 0u : rp - d.Lx;
  const uint32_t n = d.cols[items], wi = wall_items(d, items), wn = d.cols[wi], walls = min(d.Lx, 2u) * wn;
  const bool wall = rq < walls;
  const uint32_t ri = rq - walls, q = fastdiv(wall ? 0u : ri, d.divc_m[items], d.divc_l[items]);
  GridColumn o;
  o.on = rp >= d.Lx && (wall || (d.Lx > 2 && n != 0 && q < d.Lx - 2));
  const uint32_t at = wall ? (rq >= wn ? rq - wn : rq) : ri - q * n, len = column_len(wall ? wi : items);
  o.kx = !o.on ? 1u : wall ? (rq >= wn ? d.Lx : 1u) : q + 2;
  o.g = o.on ? 1 + at * len : 1u;
  o.g1 = o.on ? min(o.g + len, d.Ly / R - 1) : 0u;
  return o;
}

// One word (of R packed rows) per thread, or a pair: the shortest launch, for
// films and film sets that do not fill the GPU for long.  The masks need
// nothing of the lattice, so they are drawn before wait() -- while the previous
// launch of the stream still runs -- and what follows it is the loads, some
// forty operations and the store.
//
// Bound by latency where the launch is short: a word's eight Philox calls take
// some 2000 cycles however idle the SM is.  100 sweeps of 37x75x214 in a bulk
// field, a record every five: 0.98 ms with the draws behind the loads, 0.64 ms
// now; 1,000 sweeps of ten contact-angle films 8.2 and 6.6 ms.  LOOK: launches
// past kLookBlocks, where the arithmetic counts.
template <int R, bool MEAS, bool LOOK, class Wait, class AccOf>
__device__ __forceinline__ void update_word(const FilmDesc& d, const uint32_t* look, uint32_t* pool, uint32_t colour,
                                            uint32_t sweep, uint32_t at, bool meas, AccOf acc_of, Wait wait) {
  constexpr uint32_t B = 8 / R, kSeam = (R - 1) * B;  // the partner row's slot: the last of its group
  const uint32_t W = d.W;
  const uint32_t rp = R == 1 ? fastdiv(at, d.divw_m, d.divw_l) : at;
  const uint32_t w = R == 1 ? at - rp * W : 0u;
  const bool pair = rp < d.Lx;
  const GridColumn gc = grid_column<R>(d, 1, rp);
  const bool on = pair || gc.on;
  const uint32_t kx = pair ? rp + 1 : gc.kx, ky = pair || !on ? 1u : gc.g * R + 1;
  const uint32_t kx2 = (d.y_mode == kYGapbc) ? (d.Lx + 1 - kx) : kx, ky2 = d.Ly - R + 1;
  const bool any7 = __any_sync(0xFFFFFFFFu, on && (!d.cls[row_class(kx, d.Lx)].sym ||
                                                   (pair && !d.cls[row_class(kx2, d.Lx)].sym)));
  const uint32_t calls = w + 1 == W ? d.last_calls : 8u;
  if (LOOK) {
    wait();
    FilmCtx c;
    film_ctx(c, d, pool, colour, sweep);
    LayerSums r1, r2;
    const uint32_t valid1 = w + 1 == W ? c.last_mask : 0xFFFFFFFFu;
    uint32_t valid = valid1;
    if (R > 1) {
      valid = 0;
#pragma unroll
      for (uint32_t j = 0; j < R; j++) valid |= c.last_mask << (j * B);
    }
    if (on) update_looked_up<R, MEAS>(c, look, kx, ky, w, pair, calls, valid, valid1, meas, r1, r2);
    if (MEAS && meas) {
      __syncwarp();
      add_layer_sums(acc_of(), r1);
      add_lane_sums(acc_of(), r2);
    }
    return;
  }
  Drawn a{{0, 0, 0, 0, 0, 0, 0}}, b{{0, 0, 0, 0, 0, 0, 0}};
#pragma unroll 1
  for (uint32_t r = 0; r < 2; r++) {
    if (r ? !pair : !on) continue;
    const uint32_t k = r ? kx2 : kx, y = r ? ky2 : ky;
    Drawn x;
    draw_any<R, true>(x, any7, d.cls[row_class(k, d.Lx)], (k - 1) * d.Ly + y - 1, (k + y + 1 + colour) & 1u, w, calls,
                      d.last_mask == 0xFFFFFFFFu, W > 1, sweep, d.rk0, d.rk1);
    if (r) b = x;
    else a = x;
  }
  wait();
  // what the draws do not need is read from the descriptor only now
  FilmCtx c;
  film_ctx(c, d, pool, colour, sweep);
  LayerSums r1, r2;
  if (on) {
    const ClassDraw &cl = d.cls[row_class(kx, c.Lx)], &cl2 = d.cls[row_class(kx2, c.Lx)];
    const uint32_t valid1 = w + 1 == W ? c.last_mask : 0xFFFFFFFFu;  // one row's sites
    uint32_t valid = valid1;
    if (R > 1) {
      valid = 0;
#pragma unroll
      for (uint32_t j = 0; j < R; j++) valid |= c.last_mask << (j * B);
    }
    Hood h, g;
    fetch_rows<R>(c, kx, ky, w, h);
    if (pair) fetch_rows<R>(c, kx2, ky2, w, g);
    const Count k = count_up(h);
    const uint32_t v = h.S ^ (decide(h, k, any7, a, cl) & valid);
    store_rows<R>(c, kx, ky, w, v);
    if (MEAS && meas) r1 = word_sums(kx, k, v, h.z0, valid, bond_slots(kx, c.Lx, c.x_pbc));
    if (pair) {
      // the partner's wrap neighbour is the word just decided where the seam
      // joins one colour
      if (c.seam_same) g.yp = (g.yp & ~(valid1 << kSeam)) | (((v ^ c.neg) & valid1) << kSeam);
      const Count k2 = count_up(g);
      const uint32_t v2 = g.S ^ (decide(g, k2, any7, b, cl2) & valid);
      store_rows<R>(c, kx2, ky2, w, v2);
      if (MEAS && meas) {
        r2 = word_sums(kx2, k2, v2, g.z0, valid, bond_slots(kx2, c.Lx, c.x_pbc));
        if (c.seam_same) r2.b += seam_adjust(v, h.z0, g.S, g.z0, kSeam, c.neg, valid1);
      }
    }
  }
  if (MEAS && meas) {
    add_layer_sums(acc_of(), r1);
    add_lane_sums(acc_of(), r2);
  }
}

// The columns of a film's launch: thread `at` has word w of the rows ky, ky + 1, ...
// of a layer (packed: of groups of R rows), and decides one after another.
// Rows next to each other update opposite arrays and read each other's other
// array, so a step loads five words where a lone row loads seven, the
// addresses move by a row, and what depends on the layer is set up once.  The
// first Lx * W columns are the pairs (update_pair); kept together, they fill
// whole warps.
//
// By masks: a step's need nothing of the lattice, so the first step's are drawn
// before wait() -- while the previous launch of the stream still runs.  LOOK: by
// look-ups, every word of whatever class at one comparison per site.
//
// Bound by the integer pipes (the draws: 805 of a word's some 1000 cycles per
// warp scheduler), not by memory.  120x240x1600 (46M sites), one sweep without
// records: 42.1 us with a look-up per site and two words per thread in any
// order; by masks 38.2 us in columns of two, 40.4 in columns of four; in a bulk
// field by look-ups 40.7 and 41.4 (by seven masks 63.1).  The seven masks of the
// walls are a loop over the calls: unrolled, both mask forms together overran the
// instruction cache (1.4 stalls per issue; 41.9 us), and masks beside look-ups
// for the walls alone were slower too (39.9).  The look-ups of a full word are
// straight-line code: as a loop 48.1 us.  Columns of three or five words and
// five or seven blocks per SM were slower (by 1 to 4%; by look-ups seven blocks
// are 1% faster), and so were masks drawn two steps ahead (registers).
template <int R, bool MEAS, bool LOOK, class Wait, class AccOf>
__device__ __forceinline__ void update_columns(const FilmDesc& d, const FilmCtx& c, const uint32_t* look, uint32_t at,
                                               uint32_t items, bool meas, AccOf acc_of, Wait wait) {
  constexpr uint32_t B = 8 / R;
  const uint32_t W = c.W;
  const uint32_t rp = R == 1 ? fastdiv(at, d.divw_m, d.divw_l) : at;
  const uint32_t w = R == 1 ? at - rp * W : 0u;
  const uint32_t calls = w + 1 == W ? c.last_calls : 8u;
  const uint32_t valid1 = w + 1 == W ? c.last_mask : 0xFFFFFFFFu;  // one row's sites
  uint32_t valid = valid1;
  if (R > 1) {
    valid = 0;
#pragma unroll
    for (uint32_t j = 0; j < R; j++) valid |= c.last_mask << (j * B);
  }
  // the column: groups g .. g1 - 1 of layer kx (none for a pair's thread; an idle
  // thread's range is empty, the drawing-only step included)
  const GridColumn gc = grid_column<R>(d, items, rp);
  const bool mine = gc.on;
  const uint32_t kx = gc.kx, g = gc.g, g1 = gc.g1;
  const uint32_t ci = row_class(kx, c.Lx);
  const ClassDraw& cl = c.cls[ci];
  const bool any7 = !LOOK && __any_sync(0xFFFFFFFFu, mine && !cl.sym);
  if (rp < c.Lx) {
    if (LOOK) {
      LayerSums r1, r2;
      wait();
      update_looked_up<R, MEAS>(c, look, rp + 1, 1, w, true, calls, valid, valid1, meas, r1, r2);
      if (MEAS && meas) {
        add_lane_sums(acc_of(), r1);
        add_lane_sums(acc_of(), r2);
      }
    } else {
      update_pair<R, MEAS>(c, rp + 1, w, calls, valid, valid1, meas, acc_of, wait);
    }
    if (!MEAS) return;
  }
  LayerSums sum;
  // R = 1: pA is row ky's word in the array it updates, pB in the other; om and
  // o0 are the words of row ky - 1 (array of pA) and of pB
  uint32_t X = (kx + g * R + 2 + c.colour) & 1u;
  const uint32_t base = ((kx - 1) * c.Ly + g * R) * W + w;
  const uint32_t* pA = (X ? c.plane1 : c.plane0) + base;
  const uint32_t* pB = (X ? c.plane0 : c.plane1) + base;
  const ptrdiff_t dL = (ptrdiff_t)c.Ly * W;
  const ptrdiff_t dxm = kx > 1 ? -dL : (ptrdiff_t)(c.Lx - 1) * dL, dxp = kx < c.Lx ? dL : -(ptrdiff_t)(c.Lx - 1) * dL;
  const bool xm = kx > 1 || c.x_pbc, xp = kx < c.Lx || c.x_pbc;
  // z: array 0 meets the word before, array 1 the word after, the row's ends joined
  const int zp = w > 0 ? -1 : (int)W - 1, zn = w + 1 < W ? 1 : 1 - (int)W;
  const uint32_t sp = w > 0 ? 31u : c.pos, sn = w + 1 < W ? 31u : c.pos;
  uint32_t row = (kx - 1) * c.Ly + g * R;
  uint32_t om = 0, o0 = 0;
  // row ky's words but the second z neighbour; om and o0 the row before has held
  auto load = [&](Hood& h, uint32_t& e) {
    h.S = col_ld(c, pA, 0, X, 3);
    h.ym = om;
    h.z0 = o0;
    h.yp = col_ld(c, pA, W, X, 4);
    h.xm = xm ? col_ld(c, pA, dxm, X, 5) : 0u;
    h.xp = xp ? col_ld(c, pA, dxp, X, 6) : 0u;
    if (W > 1) e = col_ld(c, pB, X ? zn : zp, X ^ 1u, 7);
  };
  auto z_side = [&](Hood& h, uint32_t e) {
    if (W == 1) h.zs = X ? packed_next(o0, 1u, c.pos) : packed_prev(o0, 1u, c.pos);
    else h.zs = X ? shift_next(o0, 0u) | ((e & 1u) << sn) : shift_prev(o0, (e >> sp) << 31);
  };
  auto settle = [&](uint32_t n, const Hood& h, const Count& k, uint32_t v) {
    if (MEAS && meas) {
      const LayerSums r = word_sums(kx, k, v, h.z0, valid, bond_slots(kx, c.Lx, c.x_pbc));
      sum.layer = r.layer;
      sum.m += r.m;
      sum.b += r.b;
    }
    if constexpr (R > 1) {
      store_rows<R>(c, kx, n * R + 1, w, v);
    } else {
      col_st(c, pA, X, v);
      const uint32_t* p = pA + W;
      pA = pB + W;
      pB = p;
      om = o0;
      o0 = h.yp;
      X ^= 1u;
    }
  };
  auto by_masks = [&](auto general) {
    constexpr bool k7 = decltype(general)::value;
    Drawn a;
    // step n loads row n's words, draws row n + 1's masks behind the loads, and
    // decides row n; step g - 1 only draws
#pragma unroll 1
    for (uint32_t n = g - 1; n < g1; n++) {
      const bool first = n == g - 1;
      Hood h;
      uint32_t e = 0;
      if (!first) {
        if constexpr (R > 1) fetch_rows<R>(c, kx, n * R + 1, w, h);
        else load(h, e);
      }
      Drawn b;
      if (n + 1 != g1) {
        draw_any<R, true>(b, k7, cl, row, R == 1 && !first ? X ^ 1u : X, w, calls, c.last_mask == 0xFFFFFFFFu, W > 1,
                          c.sweep, c.rk0, c.rk1);
        row += R;
      }
      if (first) {
        wait();
        if (R == 1) {
          om = col_ld(c, pA, -(ptrdiff_t)W, X, 1);
          o0 = col_ld(c, pB, 0, X ^ 1u, 2);
        }
      } else {
        if constexpr (R == 1) z_side(h, e);
        const Count k = count_up(h);
        settle(n, h, k, h.S ^ (decide(h, k, k7, a, cl) & valid));
      }
      a = b;
    }
  };
  auto by_look = [&]() {
    wait();
    if (R == 1 && g < g1) {
      om = col_ld(c, pA, -(ptrdiff_t)W, X, 1);
      o0 = col_ld(c, pB, 0, X ^ 1u, 2);
    }
#pragma unroll 1
    for (uint32_t n = g; n < g1; n++) {
      Hood h;
      uint32_t e = 0;
      if constexpr (R > 1) {
        fetch_rows<R>(c, kx, n * R + 1, w, h);
      } else {
        load(h, e);
        z_side(h, e);
      }
      const Count k = count_up(h);
      const uint32_t fl = look_and_decide<R>(h, k, look, ci, cl, row, (kx + n * R + 2 + c.colour) & 1u, w, calls,
                                                            W > 1, c.sweep, c.rk0, c.rk1);
      row += R;
      settle(n, h, k, h.S ^ (fl & valid));
    }
  };
  if constexpr (LOOK) {
    by_look();
  } else {
    if (any7) by_masks(std::true_type{});
    else by_masks(std::false_type{});
  }
  if (MEAS && meas) {
    __syncwarp();
    add_layer_sums(acc_of(), sum);
  }
  wait();  // a thread without a word too: the launch must not end before its predecessor
}

}  // namespace

// Half-sweep of every film of a launch: block b handles kFilmThreads columns of
// film owner[b] (the grid has a block per entry of that table), whose descriptor is staged in shared memory.  MODE
// kUpdAccumulate: the half-sweep 1 launch of a sweep after which some film
// records; those films add their record sums into their accumulators in `part`.  MODE kUpdWriteRecord: a half-sweep 0 launch right
// after such a sweep; the last block of each film that recorded after
// `rec_done` sweeps writes that record (write_record) before its update, so
// the write overlaps the launch's other blocks.  The last block holds the
// film's ragged end, so it has the fewest words; the first ones hold the pairs.
//
// The masks are drawn before pdl_wait, from the film's sweep counter.
// advance_kernel writes that, and slab_store where a lane has swept in shared
// memory, both between chunks: the first launch of a chunk (`first`) waits
// before it reads the counter and lets its successor start only then, so every
// later launch of the chunk starts after the write.
enum : uint32_t { kUpdPlain = 0, kUpdAccumulate = 1, kUpdWriteRecord = 2 };

__device__ __forceinline__ uint32_t last_update_block(const FilmDesc& d, uint32_t items) {
  return d.upd_block_begin + update_blocks(d, items) - 1;
}

template <uint32_t MODE, bool PK, uint32_t FORM>
__global__ void __launch_bounds__(kFilmThreads, multi_min_blocks(FORM, MODE == kUpdAccumulate, PK))
update_kernel(const FilmDesc* __restrict__ films, const uint32_t* __restrict__ owner,
              uint32_t* __restrict__ pool, uint32_t colour, uint32_t k, uint32_t items,
              int64_t* __restrict__ part, int64_t* __restrict__ records, uint32_t rec_done, uint32_t first) {
  constexpr bool MEAS = MODE == kUpdAccumulate;
  constexpr uint32_t kDescWords = sizeof(FilmDesc) / 4;
  static_assert(sizeof(FilmDesc) % 16 == 0, "descriptor copied as uint4");
  __shared__ __align__(16) FilmDesc s_d;
  __shared__ int64_t s_red[MODE == kUpdWriteRecord ? kFilmThreads / 32 : 1];
  __shared__ uint32_t s_slot;
  __shared__ uint32_t s_look[kLookWords];
  if (first) pdl_wait();
  pdl_trigger();
  // owner table and descriptor are written by the host before the launch
  const uint32_t vb = blockIdx.x;
  const uint32_t f = owner[vb];  // the same for every thread of the block
  const uint4* src = reinterpret_cast<const uint4*>(films + f);
  uint4* dst = reinterpret_cast<uint4*>(&s_d);
  for (uint32_t i = threadIdx.x; i < kDescWords / 4; i += blockDim.x) dst[i] = src[i];
  __syncthreads();
  if (threadIdx.x == 0) s_d.sweep = __ldcg(&films[f].sweep);  // around L1: an earlier chunk's line may be there
  if (FORM == kFormColumnsLook || FORM == kFormWordLook) fill_look(s_look, s_d.cls);
  __syncthreads();
  const uint32_t t = s_d.sweep + k;
  if (!s_d.active || t > s_d.sweep_end || (MODE != kUpdWriteRecord && t >= s_d.sweep_end)) {
    pdl_wait();  // the launch must not end before its predecessor has
    return;
  }
  FilmCtx c;
  film_ctx(c, s_d, pool, colour, t);
  const bool meas = MEAS && measured_now(s_d, k + 1, 0);
  const FilmDesc* sd = &s_d;
  auto acc_of = [part, sd]() { return reinterpret_cast<unsigned long long*>(part + acc_offset(*sd)); };
  auto wait = [&]() { pdl_wait(); };
  if (MODE == kUpdWriteRecord && vb == last_update_block(s_d, items) && records_after(s_d, s_d.sweep, rec_done)) {
    pdl_wait();
    write_record(const_cast<FilmDesc*>(films + f), s_d, s_d.sweep, part, records, rec_done, s_red, &s_slot);
  }
  if (MODE == kUpdWriteRecord && t >= s_d.sweep_end) {
    pdl_wait();
    return;
  }
  const uint32_t at = (vb - s_d.upd_block_begin) * kFilmThreads + threadIdx.x;
  if (FORM == kFormWord || FORM == kFormWordLook) {
    constexpr bool LOOK = FORM == kFormWordLook;
    if (PK && s_d.pack == 4) update_word<4, MEAS, LOOK>(s_d, s_look, pool, colour, t, at, meas, acc_of, wait);
    else if (PK && s_d.pack == 2) update_word<2, MEAS, LOOK>(s_d, s_look, pool, colour, t, at, meas, acc_of, wait);
    else update_word<1, MEAS, LOOK>(s_d, s_look, pool, colour, t, at, meas, acc_of, wait);
  } else {
    constexpr bool LOOK = FORM == kFormColumnsLook;
    if (PK && s_d.pack == 4) update_columns<4, MEAS, LOOK>(s_d, c, s_look, at, items, meas, acc_of, wait);
    else if (PK && s_d.pack == 2) update_columns<2, MEAS, LOOK>(s_d, c, s_look, at, items, meas, acc_of, wait);
    else update_columns<1, MEAS, LOOK>(s_d, c, s_look, at, items, meas, acc_of, wait);
  }
}

// Single-film half-sweep.  The descriptor is a __grid_constant__ kernel
// parameter, so every per-film constant (round keys included) is read straight
// from the constant bank, and the sweep is known before pdl_wait.  MEAS:
// half-sweep 1 before a record, whose sums go into the film's accumulators
// acc.
template <int R, bool MEAS, uint32_t FORM>
__global__ void __launch_bounds__(kFilmThreads, film_min_blocks(R, MEAS, FORM))
update_film_kernel(const __grid_constant__ FilmDesc d, uint32_t* __restrict__ pool, uint32_t colour,
                   uint32_t sweep, uint32_t items, int64_t* __restrict__ acc) {
  __shared__ uint32_t s_look[kLookWords];
  pdl_trigger();
  if (FORM == kFormWordLook || FORM == kFormColumnsLook) {
    fill_look(s_look, d.cls);
    __syncthreads();
  }
  FilmCtx c;
  film_ctx(c, d, pool, colour, sweep);
  auto acc_of = [acc]() { return reinterpret_cast<unsigned long long*>(acc); };
  auto wait = [&]() { pdl_wait(); };
  const uint32_t at = blockIdx.x * kFilmThreads + threadIdx.x;
  if (FORM == kFormWord || FORM == kFormWordLook)
    update_word<R, MEAS, FORM == kFormWordLook>(d, s_look, pool, colour, sweep, at, MEAS, acc_of, wait);
  else update_columns<R, MEAS, FORM == kFormColumnsLook>(d, c, s_look, at, items, MEAS, acc_of, wait);
}

// ------------------------------------------------------------ measurement

namespace {

// One lattice word for measure_word, its index tested in checked builds.
struct CheckedLoad {
  __device__ __forceinline__ uint32_t operator()(const uint32_t* p, size_t idx, size_t lim, uint32_t site) const {
    return ISG_LD(p, idx, lim, site);
  }
};

}  // namespace

__global__ void __launch_bounds__(kMeasureBlock)
measure_partial_kernel(const FilmDesc* __restrict__ films, const uint32_t* __restrict__ owner,
                       const LaunchHdr* __restrict__ hdr, const uint32_t* __restrict__ pool,
                       int64_t* __restrict__ part, uint32_t done, int force) {
  __shared__ int64_t s_red[kMeasureBlock / 32];
  __shared__ int s_m[kMeasureMaxLpu];
  pdl_trigger();
  pdl_wait();
  const uint32_t nvb = hdr->meas_blocks;
  for (uint32_t vb = blockIdx.x; vb < nvb; vb += gridDim.x) {
    const FilmDesc& F = films[owner[vb]];
    if (!F.active || !measured_now(F, done, force)) continue;
    const uint32_t Lx = F.Lx, Ly = F.Ly, W = F.W, bpl = F.meas_bpl;
    if (F.meas_lpu > 1) {
      // several small layers per block: layer sums by shared atomics, one
      // bond-sum reduction; the bond sum goes to the first layer's slot
      const uint32_t* A = pool + F.spin_off;
      const uint32_t* B = A + (size_t)Lx * Ly * F.Wp;
      const uint32_t kx0 = (vb - F.meas_block_begin) * F.meas_lpu;
      const uint32_t nl = min(F.meas_lpu, Lx - kx0);
      const uint32_t per = Ly * W, total = nl * per;
      for (uint32_t i = threadIdx.x; i < nl; i += blockDim.x) s_m[i] = 0;
      __syncthreads();
      int64_t bsum = 0;
      for (uint32_t base = 0; base < total; base += blockDim.x) {
        const uint32_t it = base + threadIdx.x;
        const bool on = it < total;
        int m = 0, bb = 0;
        uint32_t l = 0xFFFFFFFFu;
        if (on) {
          l = it / per;
          const uint32_t r = it - l * per, kym1 = r / W;
          measure_word(CheckedLoad{}, A, B, F.Wp, Lx, Ly, W, F.n, F.last_mask, F.x_pbc, F.y_mode, kx0 + l, kym1,
                       r - kym1 * W, m, bb);
          bsum += bb;
        }
        const uint32_t l0 = __shfl_sync(0xFFFFFFFFu, l, 0);
        if (__all_sync(0xFFFFFFFFu, !on || l == l0)) {
          int v = m;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xFFFFFFFFu, v, o);
          if ((threadIdx.x & 31u) == 0 && l0 != 0xFFFFFFFFu) atomicAdd(&s_m[l0], v);
        } else if (on) {
          atomicAdd(&s_m[l], m);
        }
      }
      const int64_t tb = block_sum(bsum, s_red);  // its barriers also complete s_m
      for (uint32_t i = threadIdx.x; i < nl; i += blockDim.x) {
        int64_t* p = part + F.part_off + 2 * (size_t)(kx0 + i);
        p[0] = s_m[i];
        if (i != 0) p[1] = 0;
      }
      if (threadIdx.x == 0) part[F.part_off + 2 * (size_t)kx0 + 1] = tb;
      __syncthreads();  // s_m is read above before the next block clears it
      continue;
    }
    const uint32_t local = vb - F.meas_block_begin;
    const uint32_t kxm1 = local / bpl, chunk = local % bpl;
    const uint32_t Wp = F.Wp;
    const uint32_t* A = pool + F.spin_off;
    const uint32_t* B = A + (size_t)Lx * Ly * Wp;
    int64_t msum = 0, bsum = 0;
    for (uint32_t it = chunk * blockDim.x + threadIdx.x; it < Ly * W; it += bpl * blockDim.x) {
      const uint32_t kym1 = it / W, w = it % W;
      int m, bb;
      measure_word(CheckedLoad{}, A, B, Wp, Lx, Ly, W, F.n, F.last_mask, F.x_pbc, F.y_mode, kxm1, kym1, w, m, bb);
      msum += m;
      bsum += bb;
    }
    const int64_t tm = block_sum(msum, s_red);
    const int64_t tb = block_sum(bsum, s_red);
    if (threadIdx.x == 0) {
      int64_t* p = part + F.part_off + 2 * ((size_t)kxm1 * bpl + chunk);
      p[0] = tm;
      p[1] = tb;
    }
  }
}

__global__ void __launch_bounds__(kMeasureBlock)
measure_finalize_kernel(FilmDesc* __restrict__ films, const LaunchHdr* __restrict__ hdr,
                        const int64_t* __restrict__ part, int64_t* __restrict__ records, uint32_t done, int force,
                        int64_t* __restrict__ direct) {
  __shared__ int64_t s_red[kMeasureBlock / 32];
  __shared__ uint32_t s_slot;
  pdl_trigger();
  pdl_wait();
  const uint32_t nf = hdr->n_films;
  for (uint32_t f = blockIdx.x; f < nf; f += gridDim.x) {
    FilmDesc& F = films[f];
    if (!F.active || !measured_now(F, done, force)) continue;
    const uint32_t Lx = F.Lx, bpl = F.meas_bpl;
    __syncthreads();
    if (threadIdx.x == 0) s_slot = F.rec_cap ? (F.rec_next % F.rec_cap) : 0u;
    __syncthreads();
    int64_t* rec = direct ? direct : records + F.rec_off + (size_t)s_slot * (5 + Lx);
    const int64_t* p = part + F.part_off;
    int64_t M = 0, Bs = 0;
    for (uint32_t kx = threadIdx.x; kx < Lx; kx += blockDim.x) {
      int64_t m = 0;
      for (uint32_t c = 0; c < bpl; c++) {
        m += p[2 * ((size_t)kx * bpl + c)];
        Bs += p[2 * ((size_t)kx * bpl + c) + 1];
      }
      rec[5 + kx] = m;
      M += m;
    }
    const int64_t tM = block_sum(M, s_red);
    const int64_t tB = block_sum(Bs, s_red);
    if (threadIdx.x == 0) {
      rec[0] = (int64_t)F.sweep + done;
      rec[1] = tB;
      rec[2] = tM;
      rec[3] = rec[5];
      rec[4] = rec[5 + Lx - 1];
      if (!direct) F.rec_next = F.rec_next + 1;
    }
  }
}

// Records of the films that record after `done` sweeps of the chunk, from
// the per-layer sums half-sweep 1 accumulated; the accumulators are cleared
// for the next record.
__global__ void __launch_bounds__(kMeasureBlock)
record_kernel(FilmDesc* __restrict__ films, const LaunchHdr* __restrict__ hdr, int64_t* __restrict__ part,
              int64_t* __restrict__ records, uint32_t done) {
  __shared__ int64_t s_red[kMeasureBlock / 32];
  __shared__ uint32_t s_slot;
  pdl_trigger();
  pdl_wait();
  const uint32_t nf = hdr->n_films;
  for (uint32_t f = blockIdx.x; f < nf; f += gridDim.x) {
    FilmDesc& F = films[f];
    if (!F.active || !measured_now(F, done, 0)) continue;
    write_record(&F, F, F.sweep, part, records, done, s_red, &s_slot);
  }
}

__global__ void advance_kernel(FilmDesc* __restrict__ films, const LaunchHdr* __restrict__ hdr, uint32_t n_sweeps) {
  pdl_trigger();
  pdl_wait();
  for (uint32_t f = blockIdx.x * blockDim.x + threadIdx.x; f < hdr->n_films; f += gridDim.x * blockDim.x) {
    if (!films[f].active) continue;
    const uint32_t s = films[f].sweep, e = films[f].sweep_end;
    films[f].sweep = (e - s < n_sweeps) ? e : s + n_sweeps;
  }
}

// ------------------------------------------------------------- slab path

// Films held in shared memory for every sweep of a call: one CTA holds a film
// (C = 1), or a thread-block cluster of C CTAs holds it in distributed shared
// memory, CTA r layers kx - 1 in [r Lx / C, (r + 1) Lx / C).  Only a film's own
// CTAs meet between its half-sweeps, at a block or cluster barrier; films
// never wait for one another and no launch boundary falls between them.
//
// Layout.  In shared memory the two arrays of a row are sorted by colour, not
// by z parity: plane c holds what half-sweep c updates, so a word's six
// neighbour words all sit in the other plane (the wrap bonds of a same-colour
// seam apart), and rows of thin films are packed R to a word (fetch_rows'
// bit order).  A layer is G = Ly / R groups of W words.
//
// In small slabs a word's masks are drawn before the barrier (slab_film_tasks),
// which then hides behind the draws of the next half-sweep, and what follows it
// is loads from shared memory and bit logic; large ones (slab_film) draw behind
// it.
//
// Within a half-sweep no word is read that another thread writes (the
// checkerboard; a partner row's wrap neighbour comes from the register of the
// thread that has just decided it), so plain loads suffice, and the
// barrier's release/acquire orders one half-sweep's stores before the next
// one's loads.
namespace {

template <bool CL>
__device__ __forceinline__ uint32_t sld(uint32_t addr) {
  uint32_t v;
  if (CL) asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr));
  else asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}
template <bool CL>
__device__ __forceinline__ void sst(uint32_t addr, uint32_t v) {
  if (CL) asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
  else asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
// Adds to a sum: of the CTA's own, or (PEER) one that CTAs of the cluster share,
// which every add then reaches at cluster scope.
template <bool PEER>
__device__ __forceinline__ void sadd(uint32_t addr, int v) {
  if (PEER) asm volatile("red.relaxed.cluster.shared::cluster.add.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
  else asm volatile("red.relaxed.cta.shared::cta.add.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t v;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(v) : "r"(addr), "r"(rank));
  return v;
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

#ifdef ISING_CHECKED
__device__ __forceinline__ uint32_t in_layer(uint32_t idx, uint32_t lim, uint32_t site) {
  return oob(idx, lim, site) ? 0u : idx;
}
#else
__device__ __forceinline__ uint32_t in_layer(uint32_t idx, uint32_t, uint32_t) { return idx; }
#endif

// A film on its CTA; kept in shared memory, where it costs no registers.
struct Slab {
  uint32_t Lx, Ly, W, G, lw, pw;  // lw = G W words of a layer; pw: words of a local plane
  uint32_t a, nl;                 // first own layer (0-based), own layers
  uint32_t planes;                // shared address of the own planes
  const uint32_t* lp;             // address of layer k's plane 0 in its CTA (cluster window)
  const uint32_t* lm;             // address of layer k's sum in its CTA (a cluster: of the partner words' sum)
  uint32_t y_mode, x_pbc, last_mask, last_calls, pos, neg, seam_same;
  uint32_t len, cols;             // slab_column: words of a column, columns
};

// The words of word w of group g, layer kx, any group.  own: the layer is this
// CTA's, and so is every word but the x and wrap neighbours, which are found
// through the layer table.
template <bool CL, int R>
__device__ __forceinline__ void slab_fetch(const Slab& s, uint32_t c, bool own, uint32_t kx, uint32_t g, uint32_t w,
                                           Hood& h) {
  constexpr uint32_t B = 8 / R, kLow = slot_mask<R>(), kTop = kLow << (8 - B), kFirst = first_bits<R>();
  const uint32_t o = c ^ 1u, k = kx - 1, lim = s.lw;
  const uint32_t X = (kx + g * R + 2 + c) & 1u;  // parity array of the group's first row (ky = g R + 1)
  const uint32_t pb = 4 * s.pw;                    // plane stride in bytes
  const uint32_t i = in_layer(g * s.W + w, lim, 61);
  const uint32_t base = CL && !own ? s.lp[k] : s.planes + 4 * (k - s.a) * s.lw;
  const uint32_t bS = base + c * pb, bO = base + o * pb;
  auto ld = [&](uint32_t at) { return CL && !own ? sld<true>(at) : sld<false>(at); };
  h.S = ld(bS + 4 * i);
  h.z0 = ld(bO + 4 * i);
  const uint32_t km = k > 0 ? k - 1 : s.Lx - 1, kp = k + 1 < s.Lx ? k + 1 : 0u;
  const uint32_t xo = o * pb + 4 * i;
  if (CL) {
    h.xm = (k > 0 || s.x_pbc) ? sld<true>(s.lp[km] + xo) : 0u;
    h.xp = (k + 1 < s.Lx || s.x_pbc) ? sld<true>(s.lp[kp] + xo) : 0u;
  } else {
    h.xm = (k > 0 || s.x_pbc) ? sld<false>(s.planes + 4 * km * s.lw + xo) : 0u;
    h.xp = (k + 1 < s.Lx || s.x_pbc) ? sld<false>(s.planes + 4 * kp * s.lw + xo) : 0u;
  }
  // y neighbours: rows inside the packed word are its own other array's
  // (plane o), one slot over; the wrap row is array X of the mirrored layer
  const uint32_t gk = (s.y_mode == kYGapbc) ? (s.Lx - 1 - k) : k;
  const uint32_t gbase = CL ? s.lp[gk] : s.planes + 4 * gk * s.lw;
  uint32_t ym, yp;
  if (g > 0) ym = ld(bO + 4 * in_layer(i - s.W, lim, 62));
  else ym = sld<CL>(gbase + ((X + gk + s.Ly) & 1u) * pb + 4 * in_layer((s.G - 1) * s.W + w, lim, 63)) ^ s.neg;
  if (g + 1 < s.G) yp = ld(bO + 4 * in_layer(i + s.W, lim, 64));
  else yp = sld<CL>(gbase + ((X + (R - 1) + gk + 1) & 1u) * pb + 4 * in_layer(w, lim, 65)) ^ s.neg;
  if constexpr (R > 1) {
    ym = ((h.z0 << B) & ~kLow) | ((ym >> (8 - B)) & kLow);
    yp = ((h.z0 >> B) & ~kTop) | ((yp << (8 - B)) & kTop);
  }
  h.ym = ym;
  h.yp = yp;
  if (R > 1 || s.W == 1) {
    const uint32_t pr = packed_prev(h.z0, kFirst, s.pos), nx = packed_next(h.z0, kFirst, s.pos);
    // rows alternate between the arrays
    constexpr uint32_t kEven = R == 1 ? 0xFFFFFFFFu : R == 2 ? kLow : kLow | (kLow << 4);
    const uint32_t e = X ? ~kEven : kEven;  // slots whose row updates array 0
    h.zs = R == 1 ? (X ? nx : pr) : (pr & e) | (nx & ~e);
  } else if (X == 0) {
    const uint32_t pw = w > 0 ? ld(bO + 4 * in_layer(i - 1, lim, 66)) >> 31
                              : (ld(bO + 4 * in_layer(i + s.W - 1, lim, 67)) >> s.pos) & 1u;
    h.zs = shift_prev(h.z0, pw << 31);
  } else {
    const bool last = w + 1 == s.W;
    const uint32_t nw = ld(bO + 4 * in_layer(last ? i - w : i + 1, lim, 68));
    h.zs = shift_next(h.z0, 0u) | ((nw & 1u) << (last ? s.pos : 31u));
  }
}

__device__ __forceinline__ uint32_t slab_mirror(const Slab& s, uint32_t kx) {
  return s.y_mode == kYGapbc ? s.Lx + 1 - kx : kx;
}

// A thread's column: word w of the groups that the steps v0 .. v1 - 1 of layer kx
// name.  A layer's G steps are: the first group, its wrap partner (the last
// group of layer kx'), the groups 1 .. G - 2; a column is `len` steps, so that
// a first group and its partner are one thread's, in this order.  Columns that
// start with a first group come first, so that they share warps.
struct Column {
  uint32_t kx, w, v0, v1;
};

__device__ __forceinline__ Column slab_column(const Slab& s, uint32_t at) {
  Column o{s.a + 1, 0, 0, 0};
  if (at >= s.cols) return o;
  const uint32_t per = s.nl * s.W;
  uint32_t l, q = 0;
  if (at < per) {
    l = at / s.W;
    o.w = at - l * s.W;
  } else {
    // the others layer by layer, so that few warps hold a wall's layer
    const uint32_t r = at - per, n = s.cols / per - 1, m = r / s.W;
    o.w = r - m * s.W;
    l = m / n;
    q = m - l * n + 1;
  }
  o.kx = s.a + l + 1;
  o.v0 = q * s.len;
  o.v1 = min(o.v0 + s.len, s.G);
  return o;
}

// The words of interior group g of own layer kx: no wrap, no peer's own words.
template <bool CL, int R>
__device__ __forceinline__ void slab_fetch_in(const Slab& s, uint32_t c, uint32_t kx, uint32_t g, uint32_t w, Hood& h) {
  constexpr uint32_t B = 8 / R, kLow = slot_mask<R>(), kTop = kLow << (8 - B), kFirst = first_bits<R>();
  const uint32_t k = kx - 1, W = s.W, pb = 4 * s.pw, o = (c ^ 1u) * pb;
  const uint32_t X = (kx + g * R + 2 + c) & 1u;  // array of the group's first row
  const uint32_t i = 4 * in_layer(g * W + w, s.lw, 61);
  const uint32_t own = s.planes + 4 * (k - s.a) * s.lw + i;
  const uint32_t at = own + o;  // its other plane's word
  h.S = sld<false>(own + c * pb);
  h.z0 = sld<false>(at);
  const uint32_t ym = sld<false>(at - 4 * W), yp = sld<false>(at + 4 * W);
  const uint32_t km = k > 0 ? k - 1 : s.Lx - 1, kp = k + 1 < s.Lx ? k + 1 : 0u;
  h.xm = (k > 0 || s.x_pbc) ? sld<CL>(o + i + (CL ? s.lp[km] : s.planes + 4 * km * s.lw)) : 0u;
  h.xp = (k + 1 < s.Lx || s.x_pbc) ? sld<CL>(o + i + (CL ? s.lp[kp] : s.planes + 4 * kp * s.lw)) : 0u;
  if constexpr (R == 1) {
    h.ym = ym;
    h.yp = yp;
    if (W == 1) {
      h.zs = X ? packed_next(h.z0, 1u, s.pos) : packed_prev(h.z0, 1u, s.pos);
    } else if (X == 0) {
      const uint32_t e = sld<false>(w > 0 ? at - 4 : at + 4 * (W - 1));
      h.zs = shift_prev(h.z0, (e >> (w > 0 ? 31u : s.pos)) << 31);
    } else {
      const bool last = w + 1 == W;
      const uint32_t e = sld<false>(last ? at - 4 * w : at + 4);
      h.zs = shift_next(h.z0, 0u) | ((e & 1u) << (last ? s.pos : 31u));
    }
  } else {
    h.ym = ((h.z0 << B) & ~kLow) | ((ym >> (8 - B)) & kLow);
    h.yp = ((h.z0 >> B) & ~kTop) | ((yp << (8 - B)) & kTop);
    constexpr uint32_t kEven = R == 2 ? kLow : kLow | (kLow << 4);
    const uint32_t e = X ? ~kEven : kEven;  // slots whose row updates array 0
    h.zs = (packed_prev(h.z0, kFirst, s.pos) & e) | (packed_next(h.z0, kFirst, s.pos) & ~e);
  }
}

// The record of `t` completed sweeps: this CTA writes m(kx) of its own layers,
// rank 0 the totals; both are cleared for the next record (whose sums come
// after the next barrier).  On a cluster a layer's partner words, which any CTA
// may hold, have a sum of their own (s_m[Lx ..]): adds to one address from
// several CTAs have cluster scope, those of the CTA alone need not, and the two
// must not meet at one address.
template <bool CL>
__device__ __forceinline__ void slab_record(const Slab& s, const FilmDesc& d, int64_t* records, int* s_m, int* s_tot,
                                            bool rank0, uint32_t t) {
  const uint32_t i0 = blockDim.x - 1 - threadIdx.x;  // from the threads with the fewest items on
  if (i0 >= s.nl && i0 != 0) return;
  // the ring slot: this call's records before this one, from where the ring stood
  const uint32_t nth = d.rec_next + (t / d.measure_every - d.sweep / d.measure_every) - 1;
  int64_t* rec = records + d.rec_off + (size_t)(d.rec_cap ? nth % d.rec_cap : 0u) * (5 + s.Lx);
  for (uint32_t kx = s.a + i0; kx < s.a + s.nl; kx += blockDim.x) {
    int v = s_m[kx];
    s_m[kx] = 0;
    if (CL) {
      v += s_m[s.Lx + kx];
      s_m[s.Lx + kx] = 0;
    }
    rec[5 + kx] = v;
    if (kx == 0) rec[3] = v;
    if (kx == s.Lx - 1) rec[4] = v;
  }
  if (rank0 && i0 == 0) {
    rec[0] = (int64_t)t;
    rec[1] = s_tot[0];
    rec[2] = s_tot[1];
    s_tot[0] = 0;
    s_tot[1] = 0;
  }
}

template <bool CL>
__device__ __forceinline__ void slab_arrive() {
  if (CL) asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
template <bool CL>
__device__ __forceinline__ void slab_wait() {
  if (CL) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  else asm volatile("barrier.sync 0;" ::: "memory");
}

// Sets up the slab of film d (staged in shared memory): geometry, the planes
// sorted by colour and packed R rows to a word, the layer tables, zero sums.
// Every CTA's part is in place once the cluster's next barrier has passed.
template <bool CL, int R>
__device__ __forceinline__ void slab_load(const FilmDesc& d, const uint32_t* __restrict__ pool, int* s_tot,
                                          uint32_t* s_dyn, Slab& s, uint32_t C, uint32_t rank) {
  constexpr uint32_t B = 8 / R;
  if (threadIdx.x == 0) {
    s.Lx = d.Lx; s.Ly = d.Ly; s.W = d.W; s.G = d.Ly / R; s.lw = s.G * s.W;
    s.a = rank * d.Lx / C;
    s.nl = (rank + 1) * d.Lx / C - s.a;
    s.pw = (d.Lx + C - 1) / C * s.lw;
    s.y_mode = d.y_mode; s.x_pbc = d.x_pbc; s.last_mask = d.last_mask; s.last_calls = d.last_calls;
    s.pos = bitpos((d.n - 1) & 31u);
    s.neg = d.y_mode != kYPbc ? 0xFFFFFFFFu : 0u;
    s.seam_same = seam_joins_one_colour(d.Lx, d.Ly, d.y_mode);
    s.planes = smem_addr(s_dyn);
    s.lp = s_dyn + 2 * s.pw;
    s.lm = s.lp + s.Lx;
    const SlabShape sh = slab_shape(d, C, blockDim.x);
    s.len = sh.len;
    s.cols = s.nl * s.W * ((s.G + sh.len - 1) / sh.len);
  }
  __syncthreads();
  uint32_t* planes = s_dyn;
  uint32_t* lp = s_dyn + 2 * s.pw;
  uint32_t* lm = lp + s.Lx;
  int* s_m = reinterpret_cast<int*>(lm + s.Lx);
  const uint32_t* g0 = pool + d.spin_off;
  const size_t gpl = (size_t)d.Lx * d.Ly * d.W;
  for (uint32_t i = threadIdx.x; i < 2 * s.nl * s.lw; i += blockDim.x) {
    const uint32_t c = i >= s.nl * s.lw ? 1u : 0u, r = i - c * s.nl * s.lw;
    const uint32_t l = r / s.lw, q = r - l * s.lw, g = q / s.W, w = q - g * s.W;
    uint32_t v = 0;
#pragma unroll
    for (uint32_t j = 0; j < R; j++) {
      const uint32_t row = (s.a + l) * s.Ly + g * R + j;             // kx - 1 = a + l, ky - 1 = g R + j
      const uint32_t X = (s.a + l + g * R + j + 1 + c) & 1u;         // (kx + ky + 1 + c) & 1
      v |= ISG_LD(g0, X * gpl + (size_t)row * s.W + w, 2 * gpl, 77) << (j * B);
    }
    planes[c * s.pw + r] = v;
  }
  for (uint32_t k = threadIdx.x; k < s.Lx; k += blockDim.x) {
    uint32_t q = 0;
    while (q + 1 < C && (q + 1) * s.Lx / C <= k) q++;
    const uint32_t at = s.planes + 4 * (k - q * s.Lx / C) * s.lw, am = smem_addr(s_m + (CL ? s.Lx + k : k));
    lp[k] = CL ? mapa(at, q) : at;
    lm[k] = CL ? mapa(am, q) : am;
    s_m[k] = 0;
    if (CL) s_m[s.Lx + k] = 0;
  }
  if (threadIdx.x < 2) s_tot[threadIdx.x] = 0;
}

// Writes the planes back, advances the film's counters to t1, and leaves the
// shared memory free for the next film once every peer is done.
template <bool CL, int R>
__device__ __forceinline__ void slab_store(FilmDesc* Fg, const FilmDesc& d, uint32_t* __restrict__ pool,
                                           const uint32_t* planes, const Slab& s, uint32_t rank, uint32_t t1) {
  constexpr uint32_t B = 8 / R;
  uint32_t* g0 = pool + d.spin_off;
  const size_t gpl = (size_t)d.Lx * d.Ly * d.W;
  for (uint32_t i = threadIdx.x; i < 2 * s.nl * s.lw; i += blockDim.x) {
    const uint32_t c = i >= s.nl * s.lw ? 1u : 0u, r = i - c * s.nl * s.lw;
    const uint32_t l = r / s.lw, q = r - l * s.lw, g = q / s.W, w = q - g * s.W;
    const uint32_t v = planes[c * s.pw + r];
#pragma unroll
    for (uint32_t j = 0; j < R; j++) {
      const uint32_t row = (s.a + l) * s.Ly + g * R + j;
      const uint32_t X = (s.a + l + g * R + j + 1 + c) & 1u;
      ISG_ST(g0, X * gpl + (size_t)row * s.W + w, 2 * gpl, 78, R == 1 ? v : (v >> (j * B)) & slot_mask<R>());
    }
  }
  if (rank == 0 && threadIdx.x == 0) {
    Fg->sweep = t1;
    if (d.measure_every) Fg->rec_next = d.rec_next + (t1 / d.measure_every - d.sweep / d.measure_every);
  }
  // the CTA's shared memory is free for its next film once every peer is done
  slab_arrive<CL>();
  slab_wait<CL>();
}


// The sweep this call ends before.
__device__ __forceinline__ uint32_t slab_end(const FilmDesc& d, uint32_t n_sweeps) {
  return (d.sweep_end - d.sweep < n_sweeps) ? max(d.sweep_end, d.sweep) : d.sweep + n_sweeps;
}

// n_sweeps sweeps of the film of descriptor d (staged from Fg) on this CTA or
// cluster, rows packed R to a word.  Thread i has columns i, i + T, ..., each word
// decided by look-ups.
//
// For slabs of more words than threads, whose draws fill the SM by themselves
// (slab_tasks_fit), so there is no wait to hide: bound by the integer pipes at
// five warps per scheduler.  96x192x384 on a cluster of eight, per sweep: 126 us,
// in a bulk field 125; with a word's masks drawn ahead of the barrier 155 and
// 177.
template <bool CL, int R>
__device__ __forceinline__ void slab_film(FilmDesc* Fg, const FilmDesc& d, uint32_t* __restrict__ pool,
                                          int64_t* __restrict__ records, uint32_t n_sweeps, int* s_tot, uint32_t* look,
                                          uint32_t* s_dyn, Slab& s, uint32_t C, uint32_t rank) {
  constexpr uint32_t B = 8 / R, kSeam = (R - 1) * B;  // the partner row's slot: the last of its group
  fill_look(look, d.cls);  // in place once slab_load has synchronised
  slab_load<CL, R>(d, pool, s_tot, s_dyn, s, C, rank);
  int* s_m = reinterpret_cast<int*>(s_dyn + 2 * s.pw + 2 * s.Lx);
  const uint32_t tot = CL ? mapa(smem_addr(s_tot), 0) : smem_addr(s_tot);
  const uint32_t t0 = d.sweep, t1 = slab_end(d, n_sweeps);
  const uint32_t m_every = d.measure_every;
  uint32_t m_left = m_every ? m_every - t0 % m_every : 0u;  // sweeps until the next record
  slab_arrive<CL>();
  slab_wait<CL>();  // every CTA's planes and tables are in place
  uint32_t c = 0, t = t0;
#pragma unroll 1
  while (t < t1) {
    const bool meas = c == 1 && m_left == 1;
    int tb = 0, tm = 0;
#pragma unroll 1
    for (uint32_t at = threadIdx.x; at < s.cols; at += blockDim.x) {
      const Column col = slab_column(s, at);
      const uint32_t valid1 = col.w + 1 == s.W ? s.last_mask : 0xFFFFFFFFu;  // one row's sites
      uint32_t valid = valid1;
      if (R > 1) {
        valid = 0;
#pragma unroll
        for (uint32_t j = 0; j < R; j++) valid |= s.last_mask << (j * B);
      }
      // what a first group leaves for its partner: its new word and its row's other array
      uint32_t pv = 0, pz = 0;
#pragma unroll 1
      for (uint32_t v = col.v0; v < col.v1; v++) {
        const bool partner = v == 1;
        const uint32_t kx = partner ? slab_mirror(s, col.kx) : col.kx;
        const uint32_t g = v == 0 ? 0u : partner ? s.G - 1 : v - 1;
        Hood h;
        if (v >= 2) slab_fetch_in<CL, R>(s, c, kx, g, col.w, h);
        else slab_fetch<CL, R>(s, c, !partner, kx, g, col.w, h);
        // the partner's wrap neighbour is the word just decided where the seam
        // joins one colour
        const bool seam = partner && s.seam_same;
        if (seam) h.yp = (h.yp & ~(valid1 << kSeam)) | (((pv ^ s.neg) & valid1) << kSeam);
        const Count k = count_up(h);
        const uint32_t ci = row_class(kx, s.Lx);
        const uint32_t fl = look_and_decide<R, true>(h, k, look, ci, d.cls[ci], (kx - 1) * s.Ly + g * R,
                                                     (kx + g * R + 2 + c) & 1u, col.w, col.w + 1 == s.W ? s.last_calls : 8u,
                                                     s.W > 1, t, d.rk0, d.rk1);
        const uint32_t nv = h.S ^ (fl & valid);
        const uint32_t off = 4 * (c * s.pw + in_layer(g * s.W + col.w, s.lw, 70));
        if (CL && partner) sst<true>(s.lp[kx - 1] + off, nv);
        else sst<false>(s.planes + 4 * (kx - 1 - s.a) * s.lw + off, nv);
        if (meas) {
          LayerSums r = word_sums(kx, k, nv, h.z0, valid, bond_slots(kx, s.Lx, s.x_pbc));
          if (seam) r.b += seam_adjust(pv, pz, h.S, h.z0, kSeam, s.neg, valid1);
          tb += r.b;
          tm += r.m;
          if (CL && partner) sadd<true>(s.lm[kx - 1], r.m);
          else sadd<false>(smem_addr(s_m + kx - 1), r.m);
        }
        pv = nv;
        pz = h.z0;
      }
    }
    if (meas) {
      __syncwarp();
      tb = __reduce_add_sync(0xFFFFFFFFu, tb);
      tm = __reduce_add_sync(0xFFFFFFFFu, tm);
      if ((threadIdx.x & 31u) == 0) {
        sadd<CL>(tot, tb);
        sadd<CL>(tot + 4, tm);
      }
    }
    slab_arrive<CL>();
    if (c) {
      m_left = m_every ? (m_left == 1 ? m_every : m_left - 1) : 0u;
      t++;
    }
    c ^= 1u;
    slab_wait<CL>();
    if (meas) slab_record<CL>(s, d, records, s_m, s_tot, rank == 0, t);
  }
  slab_store<CL, R>(Fg, d, pool, s_dyn, s, rank, t1);
}

// ---- tasks: the draws of a half-sweep spread evenly over the threads
//
// Films of few words per CTA are bound by latency: one warp takes some 2000
// cycles for a word's eight Philox calls however idle the SM is, and a thread
// with a pair (a first group and its wrap partner's) or a warp on a wall's layer
// takes twice that while the others wait at the barrier.  So drawing and
// deciding are separate here.  Four lanes draw a word, two calls each, and
// leave its masks in shared memory, the words of a half-sweep dealt out over
// all threads; deciding reads them and is short.  The masks drawn between two
// barriers are the next half-sweep's, in a second buffer.
//
// What bounds a sweep now is two rounds of draws (500 cycles), shared memory
// loads and barriers (a cluster's 360 to 600 cycles, a block's 16 to 76).
// 1,000 sweeps of 8^3 on one CTA, a record every sweep, took 3.05 ms
// and take 2.32 ms; a call of ten sweeps of 16x48x32 97 us on one CTA, and 61 us
// on the cluster of eight that such films now get.

// What a decision needs to know of its word; plane 0 addresses.  The plane an
// address lies in changes with the colour for every word a decision reads:
// plane = phase ^ c.
struct SlabWord {
  uint32_t own, xm, xp, ym, yp;  // the word, its x and y neighbours
  uint32_t f;                    // kW* bits; 8, 9: row class; 16..: layer
  uint32_t row;                  // index of its first row, | w << 16
  uint32_t pad;
};
// X in half-sweep 0, the phases of ym and yp, the first group (ym wraps), the
// word is its row's first, last, it has an x neighbour below, above; the last
// group (yp wraps; bit 10)
enum : uint32_t { kWX = 1, kWYm = 2, kWYp = 4, kWTop = 8, kWFirst = 16, kWLast = 32, kWXm = 64, kWXp = 128, kWEnd = 1024 };

template <bool CL, int R>
__device__ __forceinline__ SlabWord slab_word(const Slab& s, uint32_t kx, uint32_t g, uint32_t w) {
  SlabWord o;
  const uint32_t k = kx - 1, W = s.W, lim = s.lw;
  auto layer = [&](uint32_t l) { return CL ? s.lp[l] : s.planes + 4 * l * s.lw; };
  const uint32_t i = in_layer(g * W + w, lim, 61), X = (kx + g * R + 2) & 1u;
  const uint32_t base = layer(k), gk = (s.y_mode == kYGapbc) ? (s.Lx - 1 - k) : k;
  o.own = base + 4 * i;
  o.xm = layer(k > 0 ? k - 1 : s.Lx - 1) + 4 * i;
  o.xp = layer(k + 1 < s.Lx ? k + 1 : 0u) + 4 * i;
  o.ym = g > 0 ? base + 4 * in_layer(i - W, lim, 62) : layer(gk) + 4 * in_layer((s.G - 1) * W + w, lim, 63);
  o.yp = g + 1 < s.G ? base + 4 * in_layer(i + W, lim, 64) : layer(gk) + 4 * in_layer(w, lim, 65);
  o.row = (k * s.Ly + g * R) | w << 16;
  // plane of the wrapped neighbour: the one that holds array X of its row
  const uint32_t pm = g > 0 ? 1u : (X + gk + s.Ly) & 1u, pp = g + 1 < s.G ? 1u : (X + (R - 1) + gk + 1) & 1u;
  o.f = X * kWX | pm * kWYm | pp * kWYp | (g == 0 ? kWTop : 0u) | (g + 1 == s.G ? kWEnd : 0u) |
        (w == 0 ? kWFirst : 0u) | (w + 1 == W ? kWLast : 0u) | row_class(kx, s.Lx) << 8 | k << 16;
  if (k > 0 || s.x_pbc) o.f |= kWXm;
  if (k + 1 < s.Lx || s.x_pbc) o.f |= kWXp;
  o.pad = 0;
  return o;
}

// The words of a decision.  ANY: the word itself may be a peer CTA's.
template <bool CL, bool ANY, int R>
__device__ __forceinline__ void slab_read(const Slab& s, const SlabWord& a, uint32_t c, uint32_t pb, Hood& h) {
  constexpr uint32_t B = 8 / R, kLow = slot_mask<R>(), kTop = kLow << (8 - B), kFirst = first_bits<R>();
  const uint32_t S = c * pb, O = pb - S, X = (a.f ^ c) & kWX;
  h.S = sld<CL && ANY>(a.own + S);
  h.z0 = sld<CL && ANY>(a.own + O);
  h.xm = (a.f & kWXm) ? sld<CL>(a.xm + O) : 0u;
  h.xp = (a.f & kWXp) ? sld<CL>(a.xp + O) : 0u;
  h.ym = sld<CL>(a.ym + ((a.f & kWYm) ? O : S));
  h.yp = sld<CL>(a.yp + ((a.f & kWYp) ? O : S));
  if constexpr (R == 1) {
    if (s.W == 1) {
      h.zs = X ? packed_next(h.z0, 1u, s.pos) : packed_prev(h.z0, 1u, s.pos);
    } else if (X) {
      const bool last = a.f & kWLast;
      const uint32_t e = sld<CL && ANY>(a.own + O + (last ? 4 - 4 * s.W : 4));
      h.zs = shift_next(h.z0, 0u) | ((e & 1u) << (last ? s.pos : 31u));
    } else {
      const bool first = a.f & kWFirst;
      const uint32_t e = sld<CL && ANY>(a.own + O + (first ? 4 * s.W - 4 : -4));
      h.zs = shift_prev(h.z0, (e >> (first ? s.pos : 31u)) << 31);
    }
  } else {
    constexpr uint32_t kEven = R == 2 ? kLow : kLow | (kLow << 4);
    const uint32_t e = X ? ~kEven : kEven;  // slots whose row updates array 0
    h.zs = (packed_prev(h.z0, kFirst, s.pos) & e) | (packed_next(h.z0, kFirst, s.pos) & ~e);
  }
  // wrap signs, and (R > 1) the rows inside the packed word
  if (a.f & kWTop) h.ym ^= s.neg;
  if (a.f & kWEnd) h.yp ^= s.neg;
  if constexpr (R > 1) {
    h.ym = ((h.z0 << B) & ~kLow) | ((h.ym >> (8 - B)) & kLow);
    h.yp = ((h.z0 >> B) & ~kTop) | ((h.yp << (8 - B)) & kTop);
  }
}

// One lane's part of a word's masks, call number c1 on: bits 8 i for call c1,
// 8 i + D for the second call.
template <int K, int D>
__device__ __forceinline__ void draw_part(Masks<K>& a, const uint32_t (&t)[K], const PhiloxRow3& p, uint32_t ca,
                                          uint32_t cb, bool second) {
  masks_zero(a);
  uint32_t u[4], v[4];
  if (second) {
    p.draw2(ca, cb, u, v);
    put_call<0>(a, t, u);
    put_call<D>(a, t, v);
  } else {
    p.draw(ca, u);
    put_call<0>(a, t, u);
  }
}

// The draws of half-sweep (c, t) into mask buffer m: three words per three-mask
// word, then seven per general one.  Words whose four parts take
// one turn of the threads are drawn by four lanes, task i being part i & 3 of
// word i >> 2; more by one lane each (no shuffles, the row's products once per
// word): a second turn of parts falls on threads that decide as well (288 packed
// words, 24x48x20 on two CTAs: 6.7 us per sweep in two turns of parts, 4.7).  me:
// the thread's first task.
template <int R>
__device__ __forceinline__ void slab_tasks(const Slab& s, const FilmDesc& d, const SlabWord* words, uint32_t n_words,
                                           uint32_t n3, uint32_t* m, uint32_t c, uint32_t t, uint32_t me) {
  constexpr uint32_t B = 8 / R;
  constexpr int D = R == 1 ? 4 : 1;
  // four lanes are the form bound by latency, and the code's main line: the other
  // way round 8^3 takes 2.326 us per sweep instead of 2.310
  if (__builtin_expect(4 * n_words > blockDim.x, 0)) {
    for (uint32_t i = me; i < (n_words + 31u & ~31u); i += blockDim.x) {  // whole warps
      const uint32_t n = min(i, n_words - 1), f = words[n].f, rw = words[n].row;
      const bool any7 = __any_sync(0xFFFFFFFFu, n >= n3);
      Drawn a;
      draw_any<R>(a, any7, d.cls[(f >> 8) & 3u], rw & 0xFFFFu, (f ^ c) & kWX, rw >> 16,
                  R == 1 && !(f & kWLast) ? 8u : s.last_calls, s.last_mask == 0xFFFFFFFFu, s.W > 1, t, d.rk0, d.rk1);
      if (i >= n_words) continue;
      if (n < n3) {
#pragma unroll
        for (int k = 0; k < 3; k++) m[3 * n + k] = a.m[4 + k];
      } else {
        uint32_t* o = m + 3 * n3 + 7 * (n - n3);
#pragma unroll
        for (int k = 0; k < 7; k++) o[k] = a.m[k];
      }
    }
    return;
  }
  const uint32_t tasks = 4 * n_words, j = threadIdx.x & 3u;
  for (uint32_t i = me; i < (tasks + 31u & ~31u); i += blockDim.x) {  // whole warps
    const uint32_t n = min(i >> 2, n_words - 1);
    const uint32_t f = words[n].f, rw = words[n].row, w = rw >> 16;
    const uint32_t ncalls = R == 1 && !(f & kWLast) ? 8u : s.last_calls;
    const uint32_t rj = R == 1 ? 0u : R == 2 ? j >> 1 : j, q = R == 1 ? j : R == 2 ? 2 * (j & 1u) : 0u;
    const bool on = q < ncalls, second = q + D < ncalls;
    const ClassDraw& cl = d.cls[(f >> 8) & 3u];
    const bool any7 = __any_sync(0xFFFFFFFFu, n >= n3);
    const PhiloxRow3 p((rw & 0xFFFFu) + rj, t, ((f ^ c) & kWX) ^ (rj & 1u), d.rk0, d.rk1);
    const uint32_t sh = rj * B + q;
    auto share = [&](uint32_t v) {
      v = on ? v << sh : 0u;
      v |= __shfl_xor_sync(0xFFFFFFFFu, v, 1);
      return v | __shfl_xor_sync(0xFFFFFFFFu, v, 2);
    };
    if (!any7) {
      Masks<3> a;
      masks_zero(a);
      const uint32_t th[3] = {cl.t[4], cl.t[5], cl.t[6]};
      if (on) draw_part<3, D>(a, th, p, 8u * w + q, 8u * w + q + D, second);
      uint32_t v = 0;
#pragma unroll
      for (int k = 0; k < 3; k++) {
        const uint32_t x = share(a.m[k]) | ((cl.alw >> (4 + k)) & 1u ? 0xFFFFFFFFu : 0u);
        if (j == k) v = x;
      }
      if (j < 3 && (i >> 2) < n_words) m[3 * n + j] = v;
    } else {
      Masks<7> a;
      masks_zero(a);
      if (on) draw_part<7, D>(a, cl.t, p, 8u * w + q, 8u * w + q + D, second);
      uint32_t lo = 0, hi = 0;
#pragma unroll
      for (int k = 0; k < 7; k++) {
        const uint32_t x = share(a.m[k]) | ((cl.alw >> k) & 1u ? 0xFFFFFFFFu : 0u);
        if (j == (k & 3)) (k < 4 ? lo : hi) = x;
      }
      if ((i >> 2) < n_words) {
        if (n >= n3) {  // general words have seven masks
          uint32_t* o = m + 3 * n3 + 7 * (n - n3);
          o[j] = lo;
          if (j < 3) o[4 + j] = hi;
        } else if (j < 3) {  // a three-mask word in such a warp
          m[3 * n + j] = hi;
        }
      }
    }
  }
}

// The sweeps of a film by tasks.  Shared memory behind the layer sums: the words
// (three-mask words, then general ones), two mask buffers, the pair list.
template <bool CL, int R>
__device__ __forceinline__ void slab_film_tasks(FilmDesc* Fg, const FilmDesc& d, uint32_t* __restrict__ pool,
                                                int64_t* __restrict__ records, uint32_t n_sweeps, int* s_tot,
                                                uint32_t* s_dyn, Slab& s, uint32_t C, uint32_t rank) {
  constexpr uint32_t B = 8 / R, kSeam = (R - 1) * B;  // the partner row's slot: the last of its group
  slab_load<CL, R>(d, pool, s_tot, s_dyn, s, C, rank);
  int* s_m = reinterpret_cast<int*>(s_dyn + 2 * s.pw + 2 * s.Lx);
  const uint32_t tot = CL ? mapa(smem_addr(s_tot), 0) : smem_addr(s_tot);
  const uint32_t per = s.nl * s.W, n_words = per * s.G;
  // 16-byte aligned: s_dyn is, and the planes and tables before are rounded up
  SlabWord* words = reinterpret_cast<SlabWord*>(s_dyn + ((2 * s.pw + (CL ? 4 : 3) * s.Lx + 3) & ~3u));
  uint16_t* job = reinterpret_cast<uint16_t*>(words + n_words);  // word of (layer, group, w), the pairs' partners included
  uint32_t* masks = reinterpret_cast<uint32_t*>(job + ((n_words + 1) & ~1u));
  slab_arrive<CL>();
  slab_wait<CL>();  // every CTA's planes and tables are in place
  // Words in order of (group, own layer, w); the last group of a pair is its
  // partner's, in layer kx'.  The general ones go to the end: a word's place is
  // the number of words of its kind before it.
  auto general = [&](uint32_t kx) { return !d.cls[row_class(kx, s.Lx)].sym; };
  auto layer_of = [&](uint32_t g, uint32_t l) {
    const uint32_t kx = s.a + l + 1;
    return g + 1 == s.G ? slab_mirror(s, kx) : kx;
  };
  uint32_t n3 = 0;
  {
    uint32_t gen_in = 0, gen_end = 0;  // general layers among the own ones, and among their mirrors
    for (uint32_t l = 0; l < s.nl; l++) {
      gen_in += general(s.a + l + 1) ? 1u : 0u;
      gen_end += general(layer_of(s.G - 1, l)) ? 1u : 0u;
    }
    n3 = n_words - (gen_in * (s.G - 1) + gen_end) * s.W;
    for (uint32_t i = threadIdx.x; i < n_words; i += blockDim.x) {
      const uint32_t g = i / per, r = i - g * per, l = r / s.W, w = r - l * s.W;
      uint32_t before = 0;  // general layers before l in this group
      for (uint32_t q = 0; q < l; q++) before += general(layer_of(g, q)) ? 1u : 0u;
      const uint32_t kx = layer_of(g, l);
      const uint32_t at = general(kx) ? n3 + (g * gen_in + before) * s.W + w
                                      : (g * (s.nl - gen_in) + l - before) * s.W + w;
      words[at] = slab_word<CL, R>(s, kx, g, w);
      job[i] = (uint16_t)at;
    }
  }
  const uint32_t mw = 3 * n3 + 7 * (n_words - n3);  // words of a mask buffer
  __syncthreads();
  const uint32_t t0 = d.sweep, t1 = slab_end(d, n_sweeps);
  const uint32_t m_every = d.measure_every;
  uint32_t m_left = m_every ? m_every - t0 % m_every : 0u;  // sweeps until the next record
  const uint32_t pb = 4 * s.pw, jobs = n_words - per;       // a pair is one job
  bool pending = false;  // a record's sums are complete, not yet written
  // The first warps decide, so the tasks start at the warp behind them: where
  // there are threads enough, deciding one half-sweep and drawing the next go on
  // side by side.
  const uint32_t busy = ((jobs + 31u) & ~31u) % blockDim.x;
  const uint32_t me = threadIdx.x >= busy ? threadIdx.x - busy : threadIdx.x + blockDim.x - busy;
  if (t0 < t1) slab_tasks<R>(s, d, words, n_words, n3, masks, 0, t0, me);
  __syncthreads();
  uint32_t c = 0, t = t0;
#pragma unroll 1
  while (t < t1) {
    const uint32_t* m = masks + c * mw;
    const bool meas = c == 1 && m_left == 1;
    int tb = 0, tm = 0;
    for (uint32_t i = threadIdx.x; i < jobs; i += blockDim.x) {
      const bool pair = i < per;
      uint32_t v0 = 0, z0 = 0;
#pragma unroll 1
      for (uint32_t r = 0; r < (pair ? 2u : 1u); r++) {
        const uint32_t n = job[r ? i + per * (s.G - 1) : i];
        const SlabWord a = words[n];
        Hood h;
        if (r) slab_read<CL, true, R>(s, a, c, pb, h);
        else slab_read<CL, false, R>(s, a, c, pb, h);
        const uint32_t valid1 = (a.f & kWLast) ? s.last_mask : 0xFFFFFFFFu;  // one row's sites
        uint32_t valid = valid1;
        if (R > 1) {
          valid = 0;
#pragma unroll
          for (uint32_t j = 0; j < R; j++) valid |= s.last_mask << (j * B);
        }
        // the partner's wrap neighbour is the word just decided where the seam
        // joins one colour
        const bool seam = r && s.seam_same;
        if (seam) h.yp = (h.yp & ~(valid1 << kSeam)) | (((v0 ^ s.neg) & valid1) << kSeam);
        const Count k = count_up(h);
        uint32_t fl;
        if (n < n3) {
          const uint32_t* q = m + 3 * n;
          fl = flips3(h.S, k, q[0], q[1], q[2]);
        } else {
          const uint32_t* q = m + 3 * n3 + 7 * (n - n3);
          const ClassDraw& cl = d.cls[(a.f >> 8) & 3u];
          const uint32_t mm[7] = {q[0], q[1], q[2], q[3], q[4], q[5], q[6]};
          fl = flips7(h.S, k, mm, cl.up, cl.frz);
        }
        const uint32_t v = h.S ^ (fl & valid);
        if (r) sst<CL>(a.own + c * pb, v);
        else sst<false>(a.own + c * pb, v);
        if (meas) {
          const uint32_t kx = (a.f >> 16) + 1;
          LayerSums x = word_sums(kx, k, v, h.z0, valid, bond_slots(kx, s.Lx, s.x_pbc));
          if (seam) x.b += seam_adjust(v0, z0, h.S, h.z0, kSeam, s.neg, valid1);
          tb += x.b;
          tm += x.m;
          if (r) sadd<CL>(s.lm[kx - 1], x.m);
          else sadd<false>(smem_addr(s_m + kx - 1), x.m);
        }
        v0 = v;
        z0 = h.z0;
      }
    }
    if (meas) {
      __syncwarp();
      tb = __reduce_add_sync(0xFFFFFFFFu, tb);
      tm = __reduce_add_sync(0xFFFFFFFFu, tm);
      if ((threadIdx.x & 31u) == 0) {
        sadd<CL>(tot, tb);
        sadd<CL>(tot + 4, tm);
      }
      pending = true;
    }
    if (c) {
      m_left = m_every ? (m_left == 1 ? m_every : m_left - 1) : 0u;
      t++;
    }
    c ^= 1u;
    __syncwarp();
    if (t < t1) slab_tasks<R>(s, d, words, n_words, n3, masks + c * mw, c, t, me);
    slab_arrive<CL>();
    slab_wait<CL>();
    if (pending && c == 0) {
      slab_record<CL>(s, d, records, s_m, s_tot, rank == 0, t);
      pending = false;
    }
  }
  slab_store<CL, R>(Fg, d, pool, s_dyn, s, rank, t1);
}

}  // namespace

// Clusters of C CTAs (CL; else C = 1: single CTAs), cluster i sweeping films
// list[n_clusters + 1 + j] for j in [list[i], list[i + 1]) one after another
// (all n_sweeps sweeps of one, then the next); list = null: cluster i sweeps
// film i.
template <bool CL, bool TASKS>
__global__ void __launch_bounds__(TASKS ? kTaskThreads : kSlabThreads, 1)
slab_kernel(FilmDesc* __restrict__ films, const uint32_t* __restrict__ list, uint32_t n_clusters,
            uint32_t* __restrict__ pool, int64_t* __restrict__ records, uint32_t n_sweeps) {
  extern __shared__ __align__(16) uint32_t s_dyn[];
  constexpr uint32_t kDescWords = sizeof(FilmDesc) / 4;
  __shared__ __align__(16) FilmDesc s_d;
  __shared__ int s_tot[2];  // {B, M} of the record being summed (rank 0's)
  __shared__ Slab s_s;
  __shared__ uint32_t s_look[TASKS ? 1 : kLookWords];
  pdl_trigger();
  pdl_wait();
  uint32_t C = 1, rank = 0;
  if (CL) {
    cg::cluster_group cl = cg::this_cluster();
    C = cl.num_blocks();
    rank = cl.block_rank();
  }
  const uint32_t ci = blockIdx.x / C;
  if (ci >= n_clusters) return;  // the same for the whole cluster
  const uint32_t j0 = list ? list[ci] : 0u, j1 = list ? list[ci + 1] : 1u;
  for (uint32_t j = j0; j < j1; j++) {
    __syncthreads();  // every thread is done with the previous film's descriptor
    FilmDesc* Fg = films + (list ? list[n_clusters + 1 + j] : ci);
    {
      const uint4* src = reinterpret_cast<const uint4*>(Fg);
      uint4* dst = reinterpret_cast<uint4*>(&s_d);
      for (uint32_t i = threadIdx.x; i < kDescWords / 4; i += blockDim.x) dst[i] = __ldcg(src + i);
    }
    __syncthreads();
    if (!s_d.active) continue;  // the same for the whole cluster
    const uint32_t R = slab_rows(s_d, C);
    if (TASKS) {
      if (R == 4) slab_film_tasks<CL, 4>(Fg, s_d, pool, records, n_sweeps, s_tot, s_dyn, s_s, C, rank);
      else if (R == 2) slab_film_tasks<CL, 2>(Fg, s_d, pool, records, n_sweeps, s_tot, s_dyn, s_s, C, rank);
      else slab_film_tasks<CL, 1>(Fg, s_d, pool, records, n_sweeps, s_tot, s_dyn, s_s, C, rank);
    } else {
      if (R == 4) slab_film<CL, 4>(Fg, s_d, pool, records, n_sweeps, s_tot, s_look, s_dyn, s_s, C, rank);
      else if (R == 2) slab_film<CL, 2>(Fg, s_d, pool, records, n_sweeps, s_tot, s_look, s_dyn, s_s, C, rank);
      else slab_film<CL, 1>(Fg, s_d, pool, records, n_sweeps, s_tot, s_look, s_dyn, s_s, C, rank);
    }
  }
}

// ------------------------------------------------------------- set-up

__global__ void init_kernel(FilmDesc F, uint32_t* __restrict__ pool, int kind, uint32_t flip_lo, int flip_all) {
  const size_t words = (size_t)F.Lx * F.Ly * F.Wp;
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 2 * words) return;
  const uint32_t X = (uint32_t)(i / words);
  const size_t rem = i % words;
  const uint32_t row = (uint32_t)(rem / F.Wp), w = (uint32_t)(rem % F.Wp);
  if (w >= F.W) {
    pool[F.spin_off + i] = 0u;
    return;
  }
  const uint32_t ky = row % F.Ly + 1;
  const bool last = (w + 1 == F.W);
  const uint32_t valid = last ? F.last_mask : 0xFFFFFFFFu;
  uint32_t word = 0;
  if (kind == 2) {
    word = 0xFFFFFFFFu;
  } else {
    const bool up_half = ky <= F.Ly / 2;
    for (uint32_t q = 0; q < 8; q++) {
      uint32_t u[4];
      philox10(row, 8u * w + q, kInitSweep, 2u | X, F.key0, F.key1, u);
      for (uint32_t t = 0; t < 4; t++) {
        bool up;
        if (kind == 0) up = u[t] < 0x80000000u;
        else up = up_half != (flip_all || u[t] < flip_lo);
        if (up) word |= 1u << (q + 8 * t);
      }
    }
  }
  pool[F.spin_off + i] = word & valid;
}

// int8 canonical order <-> packed planes, a thread per word pair: the 64 bytes
// z0 = 64 w .. 64 w + 63 of a row hold word w of both arrays, site l = 2 k and
// 2 k + 1 of either in the k-th four of them.  They move in accesses of ALIGN
// bytes (16, 4 or 1: the largest that divides both the address and Lz).  A thread's
// bytes lie side by side, so a warp's four accesses together cover 2 KiB, and
// each of them half sectors; pack and unpack of the 46M-site film take 13 to 14 us
// each where its 52 MB take 8.  A thread per site, and one per word gathering every
// other byte, took 0.16 and 0.10 ms.
template <uint32_t ALIGN>
__device__ __forceinline__ uint32_t four_bytes(const int8_t* p, uint32_t left) {
  if (ALIGN >= 4) return *reinterpret_cast<const uint32_t*>(p);
  uint32_t v = 0;
#pragma unroll
  for (uint32_t i = 0; i < 4; i++)
    if (i < left) v |= (uint32_t)(uint8_t)p[i] << (8 * i);
  return v;
}

template <uint32_t ALIGN>
__global__ void __launch_bounds__(128) pack_kernel(FilmDesc F, uint32_t* __restrict__ pool, const int8_t* __restrict__ s) {
  const size_t words = (size_t)F.Lx * F.Ly * F.W;
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= words) return;
  const size_t row = i / F.W;
  const uint32_t w = (uint32_t)(i - row * F.W), left = F.Lz - 64u * w;  // bytes from this word on
  const int8_t* p = s + row * F.Lz + 64u * w;
  uint32_t a = 0, b = 0;
#pragma unroll
  for (uint32_t q = 0; q < 4; q++) {
    if (16u * q >= left) break;
    uint32_t v[4];
    if (ALIGN == 16) {
      const uint4 x = *reinterpret_cast<const uint4*>(p + 16 * q);
      v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    } else {
#pragma unroll
      for (uint32_t j = 0; j < 4; j++)
        v[j] = 16u * q + 4u * j < left ? four_bytes<ALIGN>(p + 16 * q + 4 * j, left - 16u * q - 4u * j) : 0u;
    }
#pragma unroll
    for (uint32_t j = 0; j < 4; j++) {
      // bit 7 of each byte: its value is above 0
      const uint32_t up = ((v[j] & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) & ~v[j] & 0x80808080u;
      const uint32_t k = 4 * q + j, at = (k >> 1) + 16 * (k & 1u);
      const uint32_t e = (up >> 7) & 0x00010001u, o = (up >> 15) & 0x00010001u;
      a |= ((e | e >> 8) & 0x0101u) << at;
      b |= ((o | o >> 8) & 0x0101u) << at;
    }
  }
  pool[F.spin_off + i] = a;
  pool[F.spin_off + words + i] = b;
}

template <uint32_t ALIGN>
__global__ void __launch_bounds__(128) unpack_kernel(FilmDesc F, const uint32_t* __restrict__ pool, int8_t* __restrict__ s) {
  const size_t words = (size_t)F.Lx * F.Ly * F.W;
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= words) return;
  const size_t row = i / F.W;
  const uint32_t w = (uint32_t)(i - row * F.W), left = F.Lz - 64u * w;
  int8_t* p = s + row * F.Lz + 64u * w;
  const uint32_t a = pool[F.spin_off + i], b = pool[F.spin_off + words + i];
#pragma unroll
  for (uint32_t q = 0; q < 4; q++) {
    if (16u * q >= left) break;
    uint32_t v[4];
#pragma unroll
    for (uint32_t j = 0; j < 4; j++) {
      const uint32_t k = 4 * q + j, at = (k >> 1) + 16 * (k & 1u);
      const uint32_t x = a >> at, y = b >> at;
      const uint32_t m = (x & 1u) | (x & 0x100u) << 8 | (y & 1u) << 8 | (y & 0x100u) << 16;
      v[j] = ~(m * 0xFEu);  // 1 where the bit is set, else -1
    }
    if (ALIGN == 16) {
      *reinterpret_cast<uint4*>(p + 16 * q) = make_uint4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (uint32_t j = 0; j < 4; j++) {
        const uint32_t at = 16u * q + 4u * j;
        if (ALIGN == 4) {
          if (at < left) *reinterpret_cast<uint32_t*>(p + at) = v[j];
        } else {
#pragma unroll
          for (uint32_t t = 0; t < 4; t++)
            if (at + t < left) p[at + t] = (int8_t)(v[j] >> (8 * t));
        }
      }
    }
  }
}

// ------------------------------------------------------ host launchers

namespace {

// Launch on st with programmatic stream serialisation: the kernel may begin
// while the previous kernel of the stream is still running and orders itself
// after it with pdl_wait.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), uint32_t grid, uint32_t block, uint32_t smem, cudaStream_t st,
                       Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace

namespace {

template <uint32_t FORM>
auto update_variant(uint32_t mode, bool pack) {
  return mode == kUpdAccumulate    ? (pack ? update_kernel<kUpdAccumulate, true, FORM> : update_kernel<kUpdAccumulate, false, FORM>)
         : mode == kUpdWriteRecord ? (pack ? update_kernel<kUpdWriteRecord, true, FORM> : update_kernel<kUpdWriteRecord, false, FORM>)
                                   : (pack ? update_kernel<kUpdPlain, true, FORM> : update_kernel<kUpdPlain, false, FORM>);
}

template <bool MEAS, uint32_t FORM>
auto update_film_variant(uint32_t pack) {
  return pack == 4 ? update_film_kernel<4, MEAS, FORM>
                   : pack == 2 ? update_film_kernel<2, MEAS, FORM> : update_film_kernel<1, MEAS, FORM>;
}

template <uint32_t FORM>
auto update_film_variant(uint32_t pack, bool meas) {
  return meas ? update_film_variant<true, FORM>(pack) : update_film_variant<false, FORM>(pack);
}

}  // namespace

cudaError_t launch_update(const LaunchSet& L, uint32_t grid, uint32_t* pool, uint32_t colour, uint32_t k,
                          uint32_t items, uint32_t form, bool pack, int64_t* part, int64_t* records, bool accumulate,
                          uint32_t rec_done, bool first, cudaStream_t st) {
  if (grid == 0) return cudaSuccess;
  const uint32_t mode = accumulate && colour == 1 ? kUpdAccumulate : rec_done && colour == 0 ? kUpdWriteRecord : kUpdPlain;
  auto* kern = form == kFormColumns       ? update_variant<kFormColumns>(mode, pack)
               : form == kFormColumnsLook ? update_variant<kFormColumnsLook>(mode, pack)
               : form == kFormWordLook    ? update_variant<kFormWordLook>(mode, pack)
                                          : update_variant<kFormWord>(mode, pack);
  return launch_pdl(kern, grid, kFilmThreads, 0, st, (const FilmDesc*)L.films, (const uint32_t*)L.owner_upd,
                    pool, colour, k, items, part, records,
                    mode == kUpdWriteRecord ? rec_done : 0u, first ? 1u : 0u);
}

cudaError_t launch_update_film(const FilmDesc& d, uint32_t* pool, uint32_t colour, uint32_t sweep, uint32_t items,
                               int64_t* acc, cudaStream_t st) {
  const uint32_t grid = update_blocks(d, items);
  const bool general = !table_form(d), meas = acc != nullptr;
  auto* kern = items != 1 ? (general ? update_film_variant<kFormColumnsLook>(d.pack, meas)
                                     : update_film_variant<kFormColumns>(d.pack, meas))
               : general && grid >= kLookBlocks ? update_film_variant<kFormWordLook>(d.pack, meas)
                                                : update_film_variant<kFormWord>(d.pack, meas);
  return launch_pdl(kern, grid, kFilmThreads, 0, st, d, pool, colour, sweep, items, acc);
}

cudaError_t launch_record(const LaunchSet& L, uint32_t grid, int64_t* part, int64_t* records, uint32_t done,
                          cudaStream_t st) {
  if (grid == 0) return cudaSuccess;
  return launch_pdl(record_kernel, grid, kMeasureBlock, 0, st, L.films, (const LaunchHdr*)L.hdr, part, records,
                    done);
}

cudaError_t launch_measure(const LaunchSet& L, uint32_t grid, uint32_t fin_grid, const uint32_t* pool,
                           int64_t* part, int64_t* records, uint32_t done, int force, int64_t* direct,
                           cudaStream_t st) {
  if (grid == 0) return cudaSuccess;
  cudaError_t e = launch_pdl(measure_partial_kernel, grid, kMeasureBlock, 0, st, (const FilmDesc*)L.films,
                             (const uint32_t*)L.owner_meas, (const LaunchHdr*)L.hdr, pool, part, done, force);
  if (e != cudaSuccess) return e;
  return launch_pdl(measure_finalize_kernel, fin_grid, kMeasureBlock, 0, st, L.films, (const LaunchHdr*)L.hdr,
                    (const int64_t*)part, records, done, force, direct);
}

cudaError_t launch_advance(const LaunchSet& L, uint32_t grid, uint32_t n_sweeps, cudaStream_t st) {
  if (grid == 0 || n_sweeps == 0) return cudaSuccess;
  return launch_pdl(advance_kernel, grid, 128, 0, st, L.films, (const LaunchHdr*)L.hdr, n_sweeps);
}

cudaError_t launch_init(const FilmDesc& f, uint32_t* pool, int kind, uint32_t flip_lo, int flip_all,
                        cudaStream_t st) {
  const size_t n = 2 * (size_t)f.Lx * f.Ly * f.Wp;
  init_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(f, pool, kind, flip_lo, flip_all);
  return cudaGetLastError();
}

namespace {

// The widest access that both the spins' address and the rows' starts allow.
uint32_t spin_align(const FilmDesc& f, const int8_t* s) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(s) | f.Lz;
  return a % 16 == 0 ? 16u : a % 4 == 0 ? 4u : 1u;
}

}  // namespace

cudaError_t launch_pack(const FilmDesc& f, uint32_t* pool, const int8_t* s, cudaStream_t st) {
  const unsigned grid = (unsigned)(((size_t)f.Lx * f.Ly * f.W + 127) / 128);
  const uint32_t al = spin_align(f, s);
  if (al == 16) pack_kernel<16><<<grid, 128, 0, st>>>(f, pool, s);
  else if (al == 4) pack_kernel<4><<<grid, 128, 0, st>>>(f, pool, s);
  else pack_kernel<1><<<grid, 128, 0, st>>>(f, pool, s);
  return cudaGetLastError();
}

cudaError_t launch_unpack(const FilmDesc& f, const uint32_t* pool, int8_t* s, cudaStream_t st) {
  const unsigned grid = (unsigned)(((size_t)f.Lx * f.Ly * f.W + 127) / 128);
  const uint32_t al = spin_align(f, s);
  if (al == 16) unpack_kernel<16><<<grid, 128, 0, st>>>(f, pool, s);
  else if (al == 4) unpack_kernel<4><<<grid, 128, 0, st>>>(f, pool, s);
  else unpack_kernel<1><<<grid, 128, 0, st>>>(f, pool, s);
  return cudaGetLastError();
}

uint32_t resident_smem_bytes(const FilmDesc& d) {
  const uint64_t sites = (uint64_t)d.Lx * d.Ly * d.Lz;
  const uint64_t bytes = 4ull * (2ull * d.Lx * d.Ly * d.W + d.Lx);
  if (sites > kResidentMaxSites || bytes > kResidentMaxSmem) return 0;
  return (uint32_t)(bytes + 8ull * d.Lx);  // the layer tables beside the planes and sums
}

// Dynamic shared memory of the task form: planes, tables, words, mask buffers.
static uint64_t slab_task_bytes(const FilmDesc& d, uint32_t C) {
  const uint64_t nlm = (d.Lx + C - 1) / C, words = nlm * (d.Ly / slab_rows(d, C)) * d.W;
  bool all7 = !d.cls[0].sym;
  // a CTA's general words: its share of the walls' layers and of their mirrors
  const uint64_t gen = all7 ? words : std::min<uint64_t>(words, 2 * (words / nlm) + 2 * d.W);
  return 8ull * words + (C > 1 ? 16ull : 12ull) * d.Lx + 16 + words * sizeof(uint32_t) * 8 + 2 * ((words + 1) & ~1ull) +
         2 * 4ull * (3 * (words - gen) + 7 * gen) + 16;
}

bool slab_tasks_fit(const FilmDesc& d, uint32_t C) {
  const uint64_t words = (uint64_t)((d.Lx + C - 1) / C) * (d.Ly / slab_rows(d, C)) * d.W;
  // More words than one turn of drawing threads go to columns, whose draws then
  // fill the SM anyway and need no masks in shared memory.  Per sweep, tasks /
  // columns: 576 words per CTA (48x96x64 on eight) 8.0 / 9.1 us, 768 (32x96x64 on
  // four) 9.9 / 9.1, 1536 (on two) 19.3 / 15.3; 1224 words of two calls (64x153x10
  // on eight) 7.5 / 8.3.
  return words * slab_calls(d, slab_rows(d, C)) <= 8 * kTaskThreads && words <= 0xFFFFu && (uint64_t)d.Lx * d.Ly <= 0xFFFFu && d.W <= 0xFFFFu &&
         slab_task_bytes(d, C) <= kClusterMaxSmem;
}

uint32_t slab_dyn_bytes(const FilmDesc& d, uint32_t C, bool tasks) {
  return tasks ? (uint32_t)slab_task_bytes(d, C) : cluster_smem_bytes(d, C);
}

uint32_t cluster_smem_bytes(const FilmDesc& d, uint32_t C) {
  if (C == 0 || C > kClusterMaxSize || d.Lx < C || d.Ly < 2 || d.Wp != d.W) return 0;
  const uint64_t nlm = (d.Lx + C - 1) / C;
  const uint64_t bytes = 8ull * nlm * d.Ly * d.W + 24ull * d.Lx;
  if (bytes > kClusterMaxSmem) return 0;
  return (uint32_t)bytes;
}

uint32_t cluster_threads(const FilmDesc& d, uint32_t C, uint32_t per_sm, bool tasks) {
  const uint32_t per = std::max<uint32_t>(per_sm, 1);
  if (!tasks) return slab_shape(d, C, kSlabThreads / per / 32 * 32).threads;
  const uint64_t words = (uint64_t)((d.Lx + C - 1) / C) * (d.Ly / slab_rows(d, C)) * d.W, tmax = kTaskThreads / per / 32 * 32;
  // four lanes per word and a thread per decision, if there is room for both
  const uint64_t t = (words + 31) / 32 * 32;
  if (5 * t <= tmax) return (uint32_t)(5 * t);
  if (2 * t <= tmax) return (uint32_t)tmax;
  const uint64_t turns = (words + tmax - 1) / tmax;  // one lane per word, in equal turns
  return (uint32_t)std::min<uint64_t>(((words + turns - 1) / turns + 31) / 32 * 32, tmax);
}

namespace {

// Dynamic shared memory of a launch with per_sm CTAs per SM: at least what the
// films need, and enough that per_sm + 1 CTAs (with the kernel's static
// shared memory and the per-block reserve) do not fit in one SM.
template <typename K>
cudaError_t cluster_launch_smem(K kern, uint32_t needed, uint32_t per_sm, uint32_t* out) {
  int dev = 0, per_smp = 0, reserve = 0;
  cudaFuncAttributes fa;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&per_smp, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&reserve, cudaDevAttrReservedSharedMemoryPerBlock, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kern);
  if (e != cudaSuccess) return e;
  const uint64_t fixed = (uint64_t)fa.sharedSizeBytes + (uint64_t)reserve;
  uint64_t pad = (uint64_t)per_smp / (per_sm + 1) + 1;  // per_sm + 1 CTAs of this size overflow the SM
  pad = pad > fixed ? (pad - fixed + 127) / 128 * 128 : 0;
  uint64_t smem = std::max<uint64_t>(needed, pad);
  if (smem > kClusterMaxSmem) smem = std::max<uint64_t>(needed, kClusterMaxSmem);
  *out = (uint32_t)smem;
  return cudaSuccess;
}

using SlabKernel = void (*)(FilmDesc*, const uint32_t*, uint32_t, uint32_t*, int64_t*, uint32_t);
SlabKernel slab_variant(uint32_t C, bool tasks) {
  return C > 1 ? (tasks ? slab_kernel<true, true> : slab_kernel<true, false>)
               : (tasks ? slab_kernel<false, true> : slab_kernel<false, false>);
}

cudaError_t slab_attributes(SlabKernel kern) {
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClusterMaxSmem);
  // the whole unified L1 as shared memory, so that per_sm padded CTAs fit
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
  return e;
}

cudaLaunchConfig_t cluster_config(uint32_t grid, uint32_t C, uint32_t smem, uint32_t threads, cudaStream_t st,
                                  cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

bool slab_launch_ok(uint32_t C, uint32_t per_sm, uint32_t smem_bytes, uint32_t threads, bool tasks) {
  return C >= 1 && C <= kClusterMaxSize && per_sm >= 1 && per_sm <= kClusterMaxPerSm && smem_bytes <= kClusterMaxSmem &&
         threads && threads % 32u == 0 && threads <= (tasks ? kTaskThreads : kSlabThreads);
}

}  // namespace

int cluster_capacity(uint32_t C, uint32_t per_sm, uint32_t smem_bytes, uint32_t threads, bool tasks,
                     uint32_t* smem_launch) {
  if (!slab_launch_ok(C, per_sm, smem_bytes, threads, tasks)) return 0;
  const SlabKernel kern = slab_variant(C, tasks);
  uint32_t smem = 0;
  if (slab_attributes(kern) != cudaSuccess || cluster_launch_smem(kern, smem_bytes, per_sm, &smem) != cudaSuccess)
    return -1;
  *smem_launch = smem;
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = cluster_config(C, C, smem, threads, nullptr, attr);
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) return -1;
  return n;
}

cudaError_t launch_cluster(FilmDesc* films, const uint32_t* list, uint32_t n_clusters, uint32_t C,
                           uint32_t smem_launch, uint32_t threads, bool tasks, uint32_t* pool, int64_t* records,
                           uint32_t n_sweeps, cudaStream_t st) {
  if (n_clusters == 0 || n_sweeps == 0) return cudaSuccess;
  if (!slab_launch_ok(C, 1, smem_launch, threads, tasks)) return cudaErrorInvalidValue;
  const SlabKernel kern = slab_variant(C, tasks);
  if (C == 1)
    return launch_pdl(kern, n_clusters, threads, smem_launch, st, films, list, n_clusters, pool, records, n_sweeps);
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = cluster_config(n_clusters * C, C, smem_launch, threads, st, attr);
  return cudaLaunchKernelEx(&cfg, kern, films, list, n_clusters, pool, records, n_sweeps);
}

int read_oob_counters(unsigned long long* count, unsigned long long* first) {
#ifdef ISING_CHECKED
  if (cudaMemcpyFromSymbol(count, g_oob_count, sizeof *count) != cudaSuccess) return -1;
  if (cudaMemcpyFromSymbol(first, g_oob_first, sizeof *first) != cudaSuccess) return -1;
  return 1;
#else
  *count = 0;
  *first = 0;
  return 0;
#endif
}

int update_blocks_per_sm() {
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, update_kernel<kUpdPlain, false, kFormWord>, kFilmThreads, 0) !=
      cudaSuccess)
    return 0;
  return nb;
}

int measure_blocks_per_sm() {
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, measure_partial_kernel, kMeasureBlock, 0) != cudaSuccess)
    return 0;
  return nb;
}

}  // namespace isg
