// rewl_resolve.cuh -- the WL sweep with the 32 trials of a group decided
// together (one warp runs one walker; lane j owns trial j of the group).
//
// What bounds the sequential form (sweep_chain_body) is the chain
//     bin -> shadow of the target bin -> compare -> next bin,
// about 130 cycles a trial on one lane.  Here every lane decides its own trial
// for an assumed acceptance vector A of the trials before it, and the warp
// repeats that until the decisions reproduce A:
//     bin before trial j   = bin + sum of the accepted offsets of trials < j
//     offset of trial j    = its offset on the group's first configuration,
//                            corrected for accepted earlier trials next to it
//     visits inside the group (where they can matter): counted, see below
//     decision of trial j  = the sequential form's test on those numbers.
// Trial j's decision depends on trials < j only, so the fixed point is unique
// and is the sequential result, and every pass settles at least the first
// trial that was still wrong: at most 33 passes, whatever the data.  Measured
// on a CPU model of the walk, a group takes 2.0 - 2.7 decisions at small ln f
// (first guess included: all trials judged from the group's first bin), 4.2 on
// an 8 x 8 lattice, and 5 - 9 at ln f = 1.
//
// A pass is a chain of about 225 cycles of a lone warp (320 with counted visits),
// a group about 530 besides.  Against the sequential forms, 1000 sweeps, whole
// calls: Ising 32 x 32, 64 walkers, ln f = 2^-18 66.1 -> 15.6 ms (134 -> 32 cycles
// a trial of a walker), from ln f = 1 on 67.4 -> 47.0 ms; Potts q = 10 32 x 32, 512
// walkers 75.1 -> 20.6 ms; +-J 12^3 114 -> 24.8 ms; Ising 8 x 8 to ln f < 1e-6
// 615 -> 112 ms; and Ising 128 x 128, 4096 walkers, 200 sweeps 600 -> 169 - 186 ms,
// where issue is what bounds it (381 warp instructions a group).
//
// Visits.  ln g of a bin grows by ln f a visit, also inside the group.  For a
// trial the counts of two bins differ by at most the number of earlier trials,
// so the test on the shadows as they stood at the start of the group decides
// whenever it is clear by more than the guard band plus that many ln f.  Only
// if some trial of the group is closer are the visits counted (BinMasks), and the
// passes go on with exact shadows; a trial inside the guard band itself is then
// decided in FP64, as in the sequential form.
#pragma once
#include <cstdint>
#include <type_traits>

#include "rewl_device.cuh"
#include "rewl_layout.h"

namespace rewl {

template <int MODEL>
constexpr int kNeighbours = MODEL == kEA3 ? 6 : 4;
template <int MODEL>
constexpr int kMaxOffset = MODEL == kPotts ? 4 : (MODEL == kEA3 ? 3 : 2);  // bins one trial can move

// One trial's draw, as its lane needs it.
struct TrialDraw {
  int64_t thr;                      // ln u in units of 2^-40
  uint32_t x, xl, xr, y, yu, yd;    // the site, its columns left and right, its rows above and below
  uint32_t z, zb, zf;               // the cube: its layer, the ones behind and in front (0 in 2D)
  uint32_t pv;                      // Potts: the proposed offset
  uint32_t js;                      // +-J: bit n: bond n has J = -1
};

// Earlier trials of the group (bit i: trial i) at this trial's site and at its neighbours
// (0 right, 1 left, 2 down, 3 up, 4 behind, 5 in front).
template <int MODEL>
struct TrialHits {
  uint32_t s;
  uint32_t n[kNeighbours<MODEL>];
  __device__ __forceinline__ uint32_t all() const {
    uint32_t m = s;
#pragma unroll
    for (int k = 0; k < kNeighbours<MODEL>; ++k) m |= n[k];
    return m;
  }
};

// Site, neighbours and proposal of the draw r (all of a TrialDraw but thr).
template <int MODEL>
__device__ __forceinline__ TrialDraw place_trial(const Problem& P, const uint32_t* J, const U4& r) {
  int x, y;
  uint32_t pv;
  trial_site<MODEL>(P, r, x, y, pv);
  TrialDraw d;
  d.thr = 0;
  const uint32_t L = (uint32_t)P.L;
  d.x = (uint32_t)x;
  d.y = (uint32_t)y;
  d.xl = (x ? d.x : L) - 1u;
  d.yu = (y ? d.y : L) - 1u;
  d.xr = d.x + 1u == L ? 0u : d.x + 1u;
  d.yd = d.y + 1u == L ? 0u : d.y + 1u;
  d.z = d.zb = d.zf = d.pv = d.js = 0u;
  if constexpr (MODEL == kPotts) d.pv = pv;
  if constexpr (MODEL == kEA) {
    d.js = coupling_bit(J, P.Wr1, 0, L, d.x, d.y) | coupling_bit(J, P.Wr1, 0, L, d.xl, d.y) << 1 |
           coupling_bit(J, P.Wr1, 1, L, d.x, d.y) << 2 | coupling_bit(J, P.Wr1, 1, L, d.x, d.yu) << 3;
  }
  if constexpr (MODEL == kEA3) {
    d.z = pv;
    d.zb = pv + 1u == L ? 0u : pv + 1u;
    d.zf = (pv ? pv : L) - 1u;
    const uint32_t zo = pv * L, R = (uint32_t)P.rows;
    d.js = coupling_bit(J, P.Wr1, 0, R, d.x, zo + d.y) | coupling_bit(J, P.Wr1, 0, R, d.xl, zo + d.y) << 1 |
           coupling_bit(J, P.Wr1, 1, R, d.x, zo + d.y) << 2 | coupling_bit(J, P.Wr1, 1, R, d.x, zo + d.yu) << 3 |
           coupling_bit(J, P.Wr1, 2, R, d.x, zo + d.y) << 4 | coupling_bit(J, P.Wr1, 2, R, d.x, d.zf * L + d.y) << 5;
  }
  return d;
}

template <int MODEL>
__device__ __forceinline__ TrialDraw draw_trial(const Problem& P, const uint32_t* J, uint64_t t, int W) {
  const U4 r = philox10((uint32_t)t, (uint32_t)(t >> 32), (uint32_t)W, kTagFlip, P.seed_lo, P.seed_hi);
  TrialDraw d = place_trial<MODEL>(P, J, r);
  const float uf = __ull2float_rn(2ull * u52_bits(r.z, r.w) + 1ull) * 0x1p-53f;
  d.thr = __float2ll_rn(logf(uf) * 1099511627776.0f);
  return d;
}

// The trials at (x, y) of a group are those in row y and in column x: two tables of lane masks
// (three on the cube), zero between groups, in place of 31 shuffles with five comparisons each.
template <int MODEL>
constexpr int kHitTables = MODEL == kEA3 ? 3 : 2;  // tables of L words

template <int MODEL>
__device__ __forceinline__ TrialHits<MODEL> find_hits(uint32_t* tab, int L, const TrialDraw& d, int lane) {
  const uint32_t bit = 1u << lane, lt = bit - 1u;
  uint32_t *R = tab, *C = tab + L, *Z = tab + 2 * L;
  atomicOr(&R[d.y], bit);
  atomicOr(&C[d.x], bit);
  if constexpr (MODEL == kEA3) atomicOr(&Z[d.z], bit);
  __syncwarp();
  TrialHits<MODEL> h;
  uint32_t ry = R[d.y] & lt, cx = C[d.x] & lt;
  if constexpr (MODEL == kEA3) {
    const uint32_t cz = Z[d.z];
    h.n[4] = ry & cx & Z[d.zb];
    h.n[5] = ry & cx & Z[d.zf];
    ry &= cz;
    cx &= cz;
  }
  h.s = ry & cx;
  h.n[0] = ry & C[d.xr];
  h.n[1] = ry & C[d.xl];
  h.n[2] = R[d.yd] & cx;
  h.n[3] = R[d.yu] & cx;
  __syncwarp();
  R[d.y] = 0u;
  C[d.x] = 0u;
  if constexpr (MODEL == kEA3) Z[d.z] = 0u;
  __syncwarp();
  return h;
}

// A trial on the configuration its group starts from.
template <int MODEL>
struct TrialBase {
  uint32_t widx;  // word of the site
  uint32_t shift; // of the site in it
  uint32_t sat;   // Ising and +-J: bit n: bond n is satisfied
  uint32_t v, n[4];  // Potts: the values of the site and its neighbours
};

template <int MODEL>
__device__ __forceinline__ TrialBase<MODEL> base_of(const Problem& P, const uint32_t* lat, const TrialDraw& d) {
  const uint32_t Wr = (uint32_t)P.Wr;
  TrialBase<MODEL> b;
  if constexpr (MODEL == kPotts) {
    const uint32_t* r = lat + d.y * Wr;
    b.widx = d.y * Wr + (d.x >> 3);
    b.shift = (d.x & 7u) * 4u;
    b.v = (lat[b.widx] >> b.shift) & 15u;
    b.n[0] = (r[d.xr >> 3] >> ((d.xr & 7u) * 4u)) & 15u;
    b.n[1] = (r[d.xl >> 3] >> ((d.xl & 7u) * 4u)) & 15u;
    b.n[2] = (lat[d.yd * Wr + (d.x >> 3)] >> b.shift) & 15u;
    b.n[3] = (lat[d.yu * Wr + (d.x >> 3)] >> b.shift) & 15u;
    b.sat = 0u;
  } else {
    const uint32_t zo = MODEL == kEA3 ? d.z * (uint32_t)P.L : 0u;
    const uint32_t row = (zo + d.y) * Wr, xw = d.x >> 5;
    b.widx = row + xw;
    b.shift = d.x & 31u;
    const uint32_t c = lat[b.widx] >> b.shift;
    uint32_t diff = ((c ^ (lat[row + (d.xr >> 5)] >> (d.xr & 31u))) & 1u) |
                    ((c ^ (lat[row + (d.xl >> 5)] >> (d.xl & 31u))) & 1u) << 1 |
                    ((c ^ (lat[(zo + d.yd) * Wr + xw] >> b.shift)) & 1u) << 2 |
                    ((c ^ (lat[(zo + d.yu) * Wr + xw] >> b.shift)) & 1u) << 3;
    if constexpr (MODEL == kEA3) {
      const uint32_t L = (uint32_t)P.L;
      diff |= ((c ^ (lat[(d.zb * L + d.y) * Wr + xw] >> b.shift)) & 1u) << 4 |
              ((c ^ (lat[(d.zf * L + d.y) * Wr + xw] >> b.shift)) & 1u) << 5;
    }
    b.sat = diff ^ d.js ^ ((1u << kNeighbours<MODEL>) - 1u);
    b.v = 0u;
  }
  return b;
}

// The trial's move for given values around it: the bin offset and (Potts) the proposed value.
__device__ __forceinline__ int potts_move(uint32_t q, uint32_t pv, uint32_t v, uint32_t n0, uint32_t n1, uint32_t n2,
                                          uint32_t n3, uint32_t& nv) {
  nv = v + 1u + pv;
  if (nv >= q) nv -= q;
  return (int)(n0 == v) + (int)(n1 == v) + (int)(n2 == v) + (int)(n3 == v) - (int)(n0 == nv) - (int)(n1 == nv) -
         (int)(n2 == nv) - (int)(n3 == nv);
}

// Sums of the bin offsets of a set of trials, without the chain of a shuffle scan: the offsets are cut into bits
// (two's complement), one ballot a bit, and a sum is a few population counts.  Ising and 2D +-J: the ballots are of
// the four bonds (the offset is the number of satisfied ones minus two), added up bitwise for all lanes at once.
template <int MODEL>
struct OffsetBits {
  static constexpr int N = kMaxOffset<MODEL> > 3 ? 4 : 3;
  uint32_t b[N];
  __device__ __forceinline__ void cut(int d, uint32_t bonds) {
    if constexpr (kNeighbours<MODEL> == 4 && MODEL != kPotts) {
      const uint32_t s0 = __ballot_sync(0xffffffffu, bonds & 1u), s1 = __ballot_sync(0xffffffffu, bonds & 2u),
                     s2 = __ballot_sync(0xffffffffu, bonds & 4u), s3 = __ballot_sync(0xffffffffu, bonds & 8u);
      const uint32_t x = s0 ^ s1 ^ s2, y = (s0 & s1) | (s0 & s2) | (s1 & s2);  // count = x + s3 + 2 y
      b[0] = x ^ s3;  // count - 2 in two's complement
      b[1] = ~(y ^ (x & s3));
      b[2] = ~(y | (x & s3));
    } else {
#pragma unroll
      for (int k = 0; k < N; ++k) b[k] = __ballot_sync(0xffffffffu, (d >> k) & 1);
    }
  }
  __device__ __forceinline__ int sum(uint32_t of) const {
    int s = __popc(b[0] & of) + 2 * __popc(b[1] & of);
    if constexpr (N == 4) s += 4 * __popc(b[2] & of) - 8 * __popc(b[3] & of);
    else s -= 4 * __popc(b[2] & of);
    return s;
  }
};
// Satisfied bonds minus half of them (a byte table for three bits: half the latency of the population count).
template <int MODEL>
__device__ __forceinline__ int offset_of_bonds(uint32_t bonds) {
  if constexpr (kNeighbours<MODEL> == 4) {
    return (int)(__byte_perm(0x02010100u, 0x03020201u, bonds & 7u) & 0xffu) + (int)(bonds >> 3) - 2;
  } else {
    return __popc(bonds) - kNeighbours<MODEL> / 2;
  }
}

// While the passes are not settled the assumed bins can lie outside the window: this many unused shadow entries
// on each side make them readable (31 accepted offsets before a trial, and its own).
__host__ __device__ __forceinline__ int resolve_reach(const Problem& P) {
  return 32 * (P.model == kPotts ? kMaxOffset<kPotts> : P.model == kEA3 ? kMaxOffset<kEA3> : kMaxOffset<kIsing>);
}

// Which trials of the group end in a bin: the end bins (counted from the group's first) cut into bits, one ballot a
// bit; the lanes equal to x are those that agree in every bit.  kBinBits bits hold -16 .. 15, where nearly every
// group stays; the rest takes eight, which is exact, since the bins of one pass span at most 33 offsets (132 for
// Potts).  Against a table of lane masks in shared memory (an atomic a trial, many of them on one word): 475 -> 333
// cycles a pass.  A bit of x picks the ballot or its complement (a predicate, in place of a mask made of two shifts:
// Ising 32 x 32 from ln f = 1 on 48.4 -> 47.0 ms
// with the checks below made once a group and one population count a bond).
constexpr int kBinBits = 5;
template <int BITS>
struct BinMasks {
  uint32_t b[BITS];
  __device__ __forceinline__ explicit BinMasks(int end) {
#pragma unroll
    for (int k = 0; k < BITS; ++k) b[k] = __ballot_sync(0xffffffffu, (end >> k) & 1);
  }
  __device__ __forceinline__ uint32_t equal(int x, uint32_t m) const {  // of the lanes m
#pragma unroll
    for (int k = 0; k < BITS; ++k) m &= (x >> k) & 1 ? b[k] : ~b[k];
    return m;
  }
};

// Shared memory of one walker: shadow, configuration, row and column tables.  BYTES: the
// configuration one byte a site (the ring form: a site is then one load away, no shifts or masks; its CTAs have
// the room); else the packed words of global memory (many walkers on one SM).
struct ResolveSmem {
  int64_t* fx;     // [-reach, P.w + reach)
  uint32_t* lat;   // packed words or bytes
  uint32_t* tab;   // [producers][kHitTables][L]
};
__host__ __device__ __forceinline__ int hit_table_words(const Problem& P) { return (P.model == kEA3 ? 3 : 2) * P.L; }
template <bool BYTES>
__host__ __device__ __forceinline__ size_t resolve_walker_bytes(const Problem& P, int tables) {
  const size_t words = (size_t)(BYTES ? (P.N + 3) / 4 : P.lat_words) + (size_t)tables * hit_table_words(P);
  const size_t bins = (size_t)P.w + 2 * resolve_reach(P);
  return (bins + (bins & 1)) * 8 + (words * 4 + 15) / 16 * 16;
}
__device__ __forceinline__ ResolveSmem resolve_carve(const Problem& P, unsigned char* base, int tables) {
  ResolveSmem m;
  const int reach = resolve_reach(P), bins = P.w + 2 * reach;
  m.fx = reinterpret_cast<int64_t*>(base) + reach;
  m.tab = reinterpret_cast<uint32_t*>(base + (size_t)(bins + (bins & 1)) * 8);
  m.lat = m.tab + tables * hit_table_words(P);
  return m;
}

// State of walker W into its shared memory (and back), by the threads t = first, first + step, ...
template <bool BYTES>
__device__ __forceinline__ void resolve_load(const Problem& P, const DevState& S, const ResolveSmem& m, int W,
                                             int tables, int first, int step) {
  const int reach = resolve_reach(P);
  for (int b = first - reach; b < P.w + reach; b += step)
    m.fx[b] = b >= 0 && b < P.w ? to_fx(double_to_bits(S.lng[(size_t)W * P.w + b])) : 0;
  const uint32_t* src = S.lat + (size_t)W * P.lat_words;
  if constexpr (BYTES) {
    uint8_t* dst = reinterpret_cast<uint8_t*>(m.lat);
    for (int i = first; i < P.N; i += step) {
      const int row = i / P.L, x = i - row * P.L;
      dst[i] = P.model == kPotts ? (src[row * P.Wr + (x >> 3)] >> ((x & 7) * 4)) & 15u
                                 : (src[row * P.Wr + (x >> 5)] >> (x & 31)) & 1u;
    }
  } else {
    for (int i = first; i < P.lat_words; i += step) m.lat[i] = src[i];
  }
  for (int i = first; i < tables * hit_table_words(P); i += step) m.tab[i] = 0u;
}
template <bool BYTES>
__device__ __forceinline__ void resolve_store(const Problem& P, const DevState& S, const ResolveSmem& m, int W,
                                              int first, int step) {
  const int kx = lnf_exponent(S.lnf[W / P.m]);
  for (int b = first; b < P.w; b += step) {
    const size_t g = (size_t)W * P.w + b;
    const uint64_t v0 = double_to_bits(S.lng[g]);
    const uint32_t c = (uint32_t)((m.fx[b] - to_fx(v0)) >> (kFxBits - kx));  // visits of the bin
    if (c) {
      S.lng[g] = bits_to_double(add_pow2_repeated(v0, kx, c));
      S.H[g] += c;
    }
  }
  uint32_t* dst = S.lat + (size_t)W * P.lat_words;
  for (int i = first; i < P.lat_words; i += step) {
    if constexpr (BYTES) {
      const uint8_t* src = reinterpret_cast<const uint8_t*>(m.lat);
      const bool potts = P.model == kPotts;
      const int per = potts ? 8 : 32, row = i / P.Wr, x0 = (i - row * P.Wr) * per;
      const int n = min(per, P.L - x0), bits = potts ? 4 * n : n;
      uint32_t word = bits == 32 ? 0u : dst[i] & ~((1u << bits) - 1u);  // what lies past a row's end stays
      for (int k = 0; k < n; ++k) word |= (uint32_t)src[row * P.L + x0 + k] << (potts ? 4 * k : k);
      dst[i] = word;
    } else {
      dst[i] = m.lat[i];
    }
  }
}

// ln f from which the passes count visits from the start (2^-kCountFrom and larger): there most groups have a
// trial that needs the counts (sweeping the shadows alone first would be wasted).
constexpr int kCountFrom = 9;

// Where walker W stands: its window, bin and ln f exponent; false if it cannot be run (the same for all threads).
struct WalkerStart {
  int wstart, w, bin, kexp;
};
__device__ __forceinline__ bool walker_start(const Problem& P, const DevState& S, int W, WalkerStart& at) {
  const int a = W / P.m;
  at.wstart = S.win_start[a];
  at.w = window_width(P, S, a);
  at.bin = (S.E[W] - P.e_min) / P.e_step - at.wstart;
  at.kexp = lnf_exponent(S.lnf[a]);
  return (unsigned)at.bin < (unsigned)at.w && at.kexp != kBadLnf;
}

// ---------------------------------------------------------------------------
// Ring of draws between the producer warps of a CTA and its walker's warp: kRingBatches batches of kRingBatch
// groups, handed over a batch at a time.  The producers do all of a trial that does not depend on the walker's
// state: the draw, the byte addresses of the site and its neighbours, and which earlier trials of the group touch it:
// as masks, and where no lane has more than two such trials (all but 3% of the groups from 24 x 24 on) as two pairs
// (trial, bonds it turns), packed into one word with the Potts offset or the signs of the couplings.
// ---------------------------------------------------------------------------
constexpr int kRingBatch = 8, kRingBatches = 2, kRingGroups = kRingBatch * kRingBatches;
constexpr int kProducers = 2;
// aux: Potts offset or coupling signs | trial 1 << 6 | trial 2 << 11 | what it turns << 16 | the same of 2 << 22 |
// (some lane of the group has more than two) << 31.  Turned: bonds (Ising, +-J); Potts: neighbours, bit 4 the site.
template <int MODEL>
struct DrawRing {
  uint4 a[kRingGroups][32];  // site, right, left, down
  uint4 b[kRingGroups][32];  // up, aux, ln u (two words)
  uint32_t touched[kRingGroups];  // trials at or next to whose site a later one of the group falls
  uint2 c[MODEL == kEA3 ? kRingGroups : 1][32];  // behind, in front
  uint32_t hits[kRingGroups][1 + kNeighbours<MODEL>][32];
  uint64_t full[kRingBatches], empty[kRingBatches];
};

template <int MODEL>
__device__ __forceinline__ void produce_draws(const Problem& P, const DevState& S, DrawRing<MODEL>& R,
                                              const uint32_t* s_J, uint32_t* tab, int W, uint32_t n_att, int producer,
                                              long long wait_cycles) {
  constexpr int NB = kNeighbours<MODEL>;
  const int lane = threadIdx.x & 31;
  const uint64_t t0 = S.clock[0] * (uint64_t)P.N;
  const uint32_t n_groups = (n_att + 31u) / 32u, L = (uint32_t)P.L;
  const long long deadline = __shfl_sync(0xffffffffu, clock64(), 0) + wait_cycles;
  for (uint32_t first = 0; first < n_groups; first += kRingBatch) {
    const uint32_t bt = (first / kRingBatch) % kRingBatches, round = first / kRingGroups;
    if (round >= 1 && !mbar_wait_warp(&R.empty[bt], (round - 1) & 1u, deadline)) {
      if (lane == 0) atomicOr(S.error, 1);
      return;
    }
    for (uint32_t g = first + producer; g < min(first + kRingBatch, n_groups); g += kProducers) {
      const uint32_t sl = g % kRingGroups, i = g * 32u + (uint32_t)lane;
      TrialDraw d = draw_trial<MODEL>(P, s_J, t0 + i, W);
      const TrialHits<MODEL> h = find_hits<MODEL>(tab, P.L, d, lane);
      if (i >= n_att) d.thr = 1ll << 62;  // past the end of the launch: never accepted
      uint32_t zo = 0u;
      if constexpr (MODEL == kEA3) {
        zo = d.z * L;
        R.c[sl][lane] = make_uint2((d.zb * L + d.y) * L + d.x, (d.zf * L + d.y) * L + d.x);
      }
      const uint32_t row = (zo + d.y) * L, around = h.all(), rest = around & (around - 1u);
      const uint32_t i1 = around ? __ffs(around) - 1 : lane, i2 = rest ? __ffs(rest) - 1 : lane;
      uint32_t t1 = 0u, t2 = 0u;
#pragma unroll
      for (int k = 0; k < NB; ++k) {
        t1 |= ((h.n[k] >> i1) & 1u) << k;
        t2 |= ((h.n[k] >> i2) & 1u) << k;
      }
      constexpr uint32_t kSelf = MODEL == kPotts ? 1u << NB : (1u << NB) - 1u;
      if ((h.s >> i1) & 1u) t1 |= kSelf;
      if ((h.s >> i2) & 1u) t2 |= kSelf;
      const bool many = __any_sync(0xffffffffu, (rest & (rest - 1u)) != 0u);
      const uint32_t touched = __reduce_or_sync(0xffffffffu, around);
      if (lane == 0) R.touched[sl] = touched;
      const uint32_t aux = (MODEL == kPotts ? d.pv : d.js) | i1 << 6 | i2 << 11 | t1 << 16 | t2 << 22 |
                           (many ? 1u << 31 : 0u);
      R.a[sl][lane] = make_uint4(row + d.x, row + d.xr, row + d.xl, (zo + d.yd) * L + d.x);
      R.b[sl][lane] = make_uint4((zo + d.yu) * L + d.x, aux, (uint32_t)d.thr,
                                 (uint32_t)((uint64_t)d.thr >> 32));
      R.hits[sl][0][lane] = h.s;
#pragma unroll
      for (int k = 0; k < NB; ++k) R.hits[sl][1 + k][lane] = h.n[k];
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&R.full[bt]);
  }
}

// The walker's side of the ring.
template <int MODEL>
struct RingReader {
  DrawRing<MODEL>& R;
  uint32_t n_groups;
  long long deadline;
  int32_t* error;
  uint4 a, b;
  uint2 c;
  __device__ __forceinline__ bool fetch(uint32_t g, int lane) {  // group g into a, b, c
    const uint32_t sl = g % kRingGroups, bt = sl / kRingBatch;
    if (g % kRingBatch == 0) {
      if (!mbar_wait_warp(&R.full[bt], (g / kRingGroups) & 1u, deadline)) {
        if (lane == 0) atomicOr(error, 2);
        return false;
      }
    }
    a = R.a[sl][lane];
    b = R.b[sl][lane];
    if constexpr (MODEL == kEA3) c = R.c[sl][lane];
    return true;
  }
  __device__ __forceinline__ void release(uint32_t g, int lane) {  // after the last read of group g (and a __syncwarp)
    if (g % kRingBatch == kRingBatch - 1 && lane == 0) mbar_arrive(&R.empty[(g % kRingGroups) / kRingBatch]);
  }
};

// ---------------------------------------------------------------------------
// Runs n_att trials of walker W on one warp.  RING: trials from a DrawRing and a configuration of bytes; else the
// warp makes its own draws (s_J: couplings) and the configuration is packed.  DENSE: trials that touch one another
// from masks; else (ring only) from the two pairs, groups with more from the masks.  COUNT: visits counted in every
// group.
// ---------------------------------------------------------------------------
template <int MODEL, bool RING, bool DENSE, bool COUNT>
__device__ __forceinline__ void resolve_walker(const Problem& P, const DevState& S, const ResolveSmem& M, int W,
                                               const WalkerStart& start, uint32_t n_att, const uint32_t* s_J,
                                               RingReader<MODEL>* ring) {
  static_assert(RING || DENSE, "pairs come from the ring");
  constexpr int NB = kNeighbours<MODEL>;
  constexpr uint32_t kAll = (1u << NB) - 1u;
  const int lane = threadIdx.x & 31;
  const uint32_t bit = 1u << lane, lt = bit - 1u;
  const int w = start.w, kexp = start.kexp;
  int bin = start.bin;
  const int lsh = kFxBits - kexp;  // ln f = 2^-kexp is 2^lsh shadow units
  const uint64_t t0 = S.clock[0] * (uint64_t)P.N;
  // The shadows at the start of a group decide trial `lane` when the difference is clear by more than this; the
  // passes look at bits 24 .. 55 only (steps of 2^-16), the exact test follows where that is close.
  const int64_t clear = kGuardFx + ((int64_t)lane << lsh);
  const uint32_t clear_24 = (uint32_t)(clear >> 24) + 1u;
  uint32_t n_acc = 0, n_tie = 0, n_exact = 0;  // of this lane's trials
  const uint32_t n_groups = (n_att + 31u) / 32u;
  const uint8_t* bytes = reinterpret_cast<const uint8_t*>(M.lat);

  // the group's trials
  int64_t thr = 0;
  uint32_t touched = 0u, site = 0u, shift = 0u, sat = 0u, v0 = 0u, n0[4] = {0u, 0u, 0u, 0u}, aux = 0u;
  TrialHits<MODEL> h;
  // their decisions (A: the accepted ones) and what follows from them
  uint32_t A = 0u, v = 0u, nv = 0u;
  int d = 0, at = 0;
  int post = -1 - lane;  // the bin the lane's trial of the previous group ended in, not yet counted
  uint32_t counting = 0u;  // the lanes that had a trial in it
  OffsetBits<MODEL> off;

  // The visits of a group: the last trial of every bin adds those of all (64-bit shared atomics are
  // compare-and-swap loops: 143 cycles even alone); the others add to unused entries, without a branch.
  auto add_visits = [&](uint32_t same) {
    same &= counting;
    const uint32_t n = __popc(same);
    int64_t* f = &M.fx[(same >> lane) == 1u ? post : -1 - lane];
    if constexpr (COUNT) *f += (int64_t)n << lsh;
    else *f += (int64_t)((uint64_t)n * (1u << lsh));  // kexp >= kCountFrom: ln f is below 2^32 units
  };
  auto load_masks = [&](uint32_t g) {
    if constexpr (RING) {
      const uint32_t sl = g % kRingGroups;
      h.s = ring->R.hits[sl][0][lane];
#pragma unroll
      for (int k = 0; k < NB; ++k) h.n[k] = ring->R.hits[sl][1 + k][lane];
    }
  };
  // The trial's offset d (and its bits) given the accepted earlier trials around it.
  auto offset = [&](auto masks) {
    constexpr bool kMasks = decltype(masks)::value;
    if constexpr (MODEL == kPotts) {
      uint32_t a[4];
      if constexpr (kMasks) {
        auto last = [&](uint32_t m, uint32_t old) {  // the value the last accepted trial of m left, else `old`
          const uint32_t got = __shfl_sync(0xffffffffu, nv, m ? 31 - __clz(m) : lane);
          return m ? got : old;
        };
        v = last(A & h.s, v0);
#pragma unroll
        for (int k = 0; k < 4; ++k) a[k] = last(A & h.n[k], n0[k]);
      } else {
        // shifts and shuffles take the low five bits of their counts
        const uint32_t v1 = __shfl_sync(0xffffffffu, nv, aux >> 6), v2 = __shfl_sync(0xffffffffu, nv, aux >> 11);
        const uint32_t t1 = __funnelshift_r(A, 0u, aux >> 6) & 1u ? aux >> 16 : 0u,
                       t2 = __funnelshift_r(A, 0u, aux >> 11) & 1u ? aux >> 22 : 0u;  // the second is the later
        v = t2 & 16u ? v2 : t1 & 16u ? v1 : v0;
#pragma unroll
        for (int k = 0; k < 4; ++k) a[k] = t2 & (1u << k) ? v2 : t1 & (1u << k) ? v1 : n0[k];
      }
      d = potts_move((uint32_t)P.q, aux & 15u, v, a[0], a[1], a[2], a[3], nv);
      off.cut(d, 0u);
    } else {
      uint32_t bonds = sat;  // every accepted flip of the site turns all its bonds, one of a neighbour the bond to it
      if constexpr (kMasks) {  // a trial is at the site or at a neighbour, not at both: one count a bond
#pragma unroll
        for (int k = 0; k < NB; ++k) bonds ^= (__popc(A & (h.s ^ h.n[k])) & 1u) << k;
      } else {
        const uint32_t on1 = __funnelshift_r(A, 0u, aux >> 6) & 1u, on2 = __funnelshift_r(A, 0u, aux >> 11) & 1u;
        bonds ^= on1 * ((aux >> 16) & kAll) ^ on2 * ((aux >> 22) & kAll);
      }
      d = offset_of_bonds<MODEL>(bonds);
      off.cut(d, bonds);
    }
  };
  using Masks = std::bool_constant<DENSE>;
  // One pass: decisions B from the acceptances A, with the visits inside the group counted if BITS > 0.
  int64_t gap = 0, f_old = 0, f_new = 0;  // gap: ln g(old) - ln g(new) - ln u
  int v_old = 0, v_new = 0;
  bool inwin = true;
  auto pass = [&](auto bin_bits, bool& wide) -> uint32_t {
    constexpr int BITS = decltype(bin_bits)::value;
    const int rel = off.sum(A & lt), to = rel + d;  // bins from the group's first
    at = bin + rel;
    inwin = (unsigned)(at + d) < (unsigned)w;
    f_old = M.fx[at];
    f_new = M.fx[at + d];
    gap = f_old - f_new - thr;
    if constexpr (BITS > 0) {
      const int end = (A & bit) ? to : rel;
      const BinMasks<BITS> ends(end);
      // the bins asked for are at most kMaxOffset further than the end bins
      constexpr uint32_t kFar = kMaxOffset<MODEL>;
      if constexpr (BITS < 8) wide = (uint32_t)end + (1u << (BITS - 1)) - kFar >= (1u << BITS) - 2u * kFar;
      v_old = __popc(ends.equal(rel, lt));
      v_new = __popc(ends.equal(to, lt));
      gap += (int64_t)(v_old - v_new) << lsh;
    }
    return __ballot_sync(0xffffffffu, inwin && gap >= 0);
  };
  // Decides the group whatever it holds, starting from A.
  auto settle = [&](uint32_t g) {
    uint32_t fixed = 0u, value = 0u;  // trials decided in FP64, and their decisions
    if constexpr (!DENSE) load_masks(g);
    while (true) {
      bool again, wide;
      do {
        const uint32_t was = nv;
        offset(std::true_type{});
        const uint32_t B = (pass(std::integral_constant<int, 8>{}, wide) & ~fixed) | value;
        again = B != A || (MODEL == kPotts && __any_sync(0xffffffffu, nv != was));
        A = B;
      } while (again);
      const uint32_t near = __ballot_sync(0xffffffffu, d != 0 && inwin &&
                                                           (uint64_t)(gap + kGuardFx) <= (uint64_t)(2 * kGuardFx)) & ~fixed;
      if (near == 0u) break;
      // the first trial inside the guard band: all before it are settled, so its numbers are final
      const int f = __ffs(near) - 1;
      bool yes = false;
      if (lane == f) {
        const uint64_t t = t0 + (uint64_t)g * 32u + (uint32_t)lane;
        const U4 r = philox10((uint32_t)t, (uint32_t)(t >> 32), (uint32_t)W, kTagFlip, P.seed_lo, P.seed_hi);
        uint64_t ties = 0;
        yes = exact_accept_fx(S, P, W, kexp, at, f_old + ((int64_t)v_old << lsh), at + d,
                              f_new + ((int64_t)v_new << lsh), u52_bits(r.z, r.w), ties);
        n_tie += (uint32_t)ties;
        ++n_exact;
      }
      fixed |= 1u << f;
      value |= __ballot_sync(0xffffffffu, yes);
      A = (A & ~(1u << f)) | (value & (1u << f));
    }
  };
  // The group's moves; those on one site compose (XOR), trials not accepted change nothing.
  auto commit = [&](uint32_t g) {
    const bool acc = (A & bit) != 0u;
    atomicXor(&M.lat[site], (acc ? (MODEL == kPotts ? v ^ nv : 1u) : 0u) << shift);
    post = acc ? at + d : at;
    counting = n_att - g * 32u >= 32u ? 0xffffffffu : (1u << (n_att - g * 32u)) - 1u;
    // the sum does not wait for `post`; with own draws (bound by issue) and with Potts' four bits a shuffle is less
    if constexpr (RING && MODEL != kPotts) bin += off.sum(A);
    else bin = __shfl_sync(0xffffffffu, post, 31);
    n_acc += acc;
    __syncwarp();
    if constexpr (RING) ring->release(g, lane);
  };

  if constexpr (RING)
    if (n_groups > 0 && !ring->fetch(0, lane)) {
      if (lane == 0) S.status[W] = kWalkerTimedOut;
      return;
    }
  // A branch around code costs a lone warp about 50 cycles, leaving a loop 10 - 30: what is rare leaves the inner
  // loop, what is short is done without asking.
  for (uint32_t g = 0; g < n_groups;) {
    uint32_t leave = 0u;  // not 0: the group needs more than the inner loop does
    bool stop = false;
    for (; g < n_groups; ++g) {
      const uint32_t same = __match_any_sync(0xffffffffu, post);
      // ---- the group's trials on the configuration as it stands
      if constexpr (RING) {
        const uint4 a = ring->a, b = ring->b;
        uint32_t c = bytes[a.x], n[NB];
        n[0] = bytes[a.y], n[1] = bytes[a.z], n[2] = bytes[a.w], n[3] = bytes[b.x];
        if constexpr (MODEL == kEA3) n[4] = bytes[ring->c.x], n[5] = bytes[ring->c.y];
        site = a.x >> 2;
        shift = (a.x & 3u) * 8u;
        aux = b.y;
        thr = (int64_t)((uint64_t)b.z | (uint64_t)b.w << 32);
        touched = ring->R.touched[g % kRingGroups];
        if constexpr (DENSE) load_masks(g);
        if (g + 1 < n_groups && !ring->fetch(g + 1, lane)) {
          stop = true;
          break;
        }
        if constexpr (MODEL == kPotts) {
          v0 = c;
#pragma unroll
          for (int k = 0; k < 4; ++k) n0[k] = n[k];
        } else {
          uint32_t nn = n[0] | n[1] << 1 | n[2] << 2 | n[3] << 3;
          if constexpr (MODEL == kEA3) nn |= n[4] << 4 | n[5] << 5;
          sat = (nn ^ (0u - c) ^ aux ^ kAll) & kAll;
        }
      } else {
        const uint32_t i = g * 32u + (uint32_t)lane;
        const TrialDraw t = draw_trial<MODEL>(P, s_J, t0 + i, W);
        h = find_hits<MODEL>(M.tab, P.L, t, lane);
        touched = __reduce_or_sync(0xffffffffu, h.all());
        thr = i < n_att ? t.thr : 1ll << 62;  // past the end of the launch: never accepted
        const TrialBase<MODEL> b0 = base_of<MODEL>(P, M.lat, t);
        add_visits(same);
        __syncwarp();
        site = b0.widx;
        shift = b0.shift;
        sat = b0.sat;
        aux = t.pv;
        if constexpr (MODEL == kPotts) {
          v0 = b0.v;
#pragma unroll
          for (int k = 0; k < 4; ++k) n0[k] = b0.n[k];
        }
      }
      v = v0;
      if constexpr (MODEL == kPotts) d = potts_move((uint32_t)P.q, aux & 15u, v0, n0[0], n0[1], n0[2], n0[3], nv);
      else d = offset_of_bonds<MODEL>(sat);

      // ---- first guess: every trial judged from the group's first bin
      at = bin;  // the bin the trial starts from, under A
      inwin = (unsigned)(at + d) < (unsigned)w;
      gap = M.fx[at] - M.fx[at + d] - thr;  // ln g(old) - ln g(new) - ln u on the shadows
      if constexpr (RING) {  // the visits of the previous group, beside the guess, which can do without them
        __syncwarp();
        add_visits(same);
      }
      A = __ballot_sync(0xffffffffu, inwin && gap >= 0);
      if constexpr (RING) __syncwarp();
      // a trial this close to the line is told by `settle` alone: without counted visits, closer than one ln f for
      // every earlier trial
      const uint32_t margin = COUNT ? 1u : clear_24;
      auto too_close = [&](bool or_else) {
        return __ballot_sync(0xffffffffu, or_else || (inwin && (uint32_t)(gap >> 24) + margin < 2u * margin + 1u));
      };
      bool again = true, wide = false;
      if constexpr (!RING) off.cut(d, sat);
      if constexpr (!RING && !COUNT) {
        leave = too_close(false);
        // a guess without a move or a touched neighbourhood is the fixed point
        again = __any_sync(0xffffffffu, (A & bit) != 0u && (d != 0 || (touched & bit) != 0u));
      }
      while (again) {
        // The offsets, for the accepted trials that touch others.  The passes that leave those alone need no new ones;
        // where a group takes two passes, asking costs as much as that saves (the ring form at small ln f).
        constexpr bool kEachPass = RING && !COUNT;
        const uint32_t was = nv, by = A & touched;
        if (RING || touched) offset(Masks{});
        const bool moved = MODEL == kPotts && __any_sync(0xffffffffu, nv != was);  // proposed values others may build on
        do {
          const uint32_t B = pass(std::integral_constant<int, COUNT ? kBinBits : 0>{}, wide);
          if constexpr (!COUNT) leave = too_close(false);
          again = B != A;
          A = B;
        } while (!kEachPass && again && (A & touched) == by);
        again = again || moved;
      }
      // With counted visits (many passes) the checks are made once, of the settled pass: bins that kBinBits do not
      // hold make a pass's decisions wrong, but still depend on the trials before alone, so the passes end.
      if constexpr (COUNT) leave = too_close(wide);
      if constexpr (!DENSE) leave |= aux >> 31;
      if (leave != 0u) break;
      commit(g);
    }
    if (stop) {  // told from out here: a store where the wait runs out costs the loop up to 5% (its registers)
      if (lane == 0) S.status[W] = kWalkerTimedOut;
      add_visits(__match_any_sync(0xffffffffu, post));
      counting = 0u;
      break;
    }
    if (g < n_groups) {
      // without counted visits: is it closer than the earlier trials' visits can make up for?
      const bool far = !COUNT && (DENSE || !(aux >> 31)) &&
                       !__any_sync(0xffffffffu, d != 0 && inwin && (uint64_t)(gap + clear) <= (uint64_t)(2 * clear));
      if (!far) settle(g);
      commit(g);
      ++g;
    }
  }
  add_visits(__match_any_sync(0xffffffffu, post));

  for (int o = 16; o; o >>= 1) {
    n_acc += __shfl_xor_sync(0xffffffffu, n_acc, o);
    n_tie += __shfl_xor_sync(0xffffffffu, n_tie, o);
    n_exact += __shfl_xor_sync(0xffffffffu, n_exact, o);
  }
  if (lane == 0) {
    S.E[W] = P.e_min + (start.wstart + bin) * P.e_step;
    S.wl_accept[W] += n_acc;
    S.near_ties[W] += n_tie;
    S.exact_tests[W] += n_exact;
  }
}

// Lattices from this many sites on take the pairs: below, more than a tenth of the groups have a trial that three
// earlier ones touch, and the masks cost a pass 45 cycles more.
constexpr int kPairSites = 400;

// Many walkers: one warp a walker, several of them in a CTA, draws made by the same warp.
template <int MODEL>
__device__ __forceinline__ void sweep_resolve_body(const Problem& P, const DevState& S, uint32_t n_att,
                                                   const int32_t* wids, int nloc) {
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t* s_J = reinterpret_cast<uint32_t*>(smem);
  const size_t j_bytes = MODEL == kEA || MODEL == kEA3 ? ((size_t)P.j_words * 4 + 15) / 16 * 16 : 0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if constexpr (MODEL == kEA || MODEL == kEA3) {
    for (int i = threadIdx.x; i < P.j_words; i += blockDim.x) s_J[i] = S.J[i];
    __syncthreads();
  }
  if (warp >= nloc) return;
  const ResolveSmem M = resolve_carve(P, smem + j_bytes + (size_t)warp * resolve_walker_bytes<false>(P, 1), 1);
  const int W = wids[warp];
  WalkerStart start;
  if (!walker_start(P, S, W, start)) {
    if (lane == 0) S.status[W] = kWalkerBadInput;
    return;
  }
  resolve_load<false>(P, S, M, W, 1, lane, 32);
  __syncwarp();
  if (start.kexp < kCountFrom) resolve_walker<MODEL, false, true, true>(P, S, M, W, start, n_att, s_J, nullptr);
  else resolve_walker<MODEL, false, true, false>(P, S, M, W, start, n_att, s_J, nullptr);
  __syncwarp();
  resolve_store<false>(P, S, M, W, lane, 32);
}

// Few walkers: one walker a CTA, its draws made by kProducers more warps.
constexpr int kRingThreads = 32 * (1 + kProducers);
template <int MODEL>
__device__ __forceinline__ void sweep_resolve_ring_body(const Problem& P, const DevState& S, uint32_t n_att, int W,
                                                        long long wait_cycles) {
  extern __shared__ __align__(16) unsigned char smem[];
  DrawRing<MODEL>& R = *reinterpret_cast<DrawRing<MODEL>*>(smem);
  uint32_t* s_J = reinterpret_cast<uint32_t*>(smem + (sizeof(DrawRing<MODEL>) + 15) / 16 * 16);
  const size_t j_bytes = MODEL == kEA || MODEL == kEA3 ? ((size_t)P.j_words * 4 + 15) / 16 * 16 : 0;
  const ResolveSmem M = resolve_carve(P, reinterpret_cast<unsigned char*>(s_J) + j_bytes, kProducers);
  const int warp = threadIdx.x >> 5;
  WalkerStart start;
  if (!walker_start(P, S, W, start)) {  // the whole CTA leaves
    if (threadIdx.x == 0) S.status[W] = kWalkerBadInput;
    return;
  }
  if constexpr (MODEL == kEA || MODEL == kEA3)
    for (int i = threadIdx.x; i < P.j_words; i += blockDim.x) s_J[i] = S.J[i];
  resolve_load<true>(P, S, M, W, kProducers, threadIdx.x, blockDim.x);
  if (threadIdx.x == 0)
    for (int k = 0; k < kRingBatches; ++k) {
      mbar_init(&R.full[k], kProducers);
      mbar_init(&R.empty[k], 1);
    }
  __syncthreads();
  if (warp == 0) {
    RingReader<MODEL> ring{R, (n_att + 31u) / 32u, __shfl_sync(0xffffffffu, clock64(), 0) + wait_cycles, S.error};
    const bool count = start.kexp < kCountFrom;
    if (P.N < kPairSites) {
      if (count) resolve_walker<MODEL, true, true, true>(P, S, M, W, start, n_att, s_J, &ring);
      else resolve_walker<MODEL, true, true, false>(P, S, M, W, start, n_att, s_J, &ring);
    } else {
      if (count) resolve_walker<MODEL, true, false, true>(P, S, M, W, start, n_att, s_J, &ring);
      else resolve_walker<MODEL, true, false, false>(P, S, M, W, start, n_att, s_J, &ring);
    }
  } else {
    produce_draws<MODEL>(P, S, R, s_J, M.tab + (warp - 1) * hit_table_words(P), W, n_att, warp - 1, wait_cycles);
  }
  __syncthreads();
  resolve_store<true>(P, S, M, W, threadIdx.x, blockDim.x);
}

__host__ __forceinline__ size_t resolve_smem_bytes(const Problem& P, int wpb, bool ring) {
  const size_t j = P.model == kEA || P.model == kEA3 ? ((size_t)P.j_words * 4 + 15) / 16 * 16 : 0;
  if (!ring) return j + (size_t)wpb * resolve_walker_bytes<false>(P, 1);
  const size_t r = P.model == kEA3 ? sizeof(DrawRing<kEA3>) : sizeof(DrawRing<kIsing>);
  return (r + 15) / 16 * 16 + j + resolve_walker_bytes<true>(P, kProducers);
}

}  // namespace rewl
