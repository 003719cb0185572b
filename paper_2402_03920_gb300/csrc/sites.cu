// SITES packing: the paper's own multi-site coding with its daemon-bit
// Metropolis rule (Sec. 2.1 and 2.1.1, Appendices B and C), for equal
// couplings k_tau = k.  A 32-bit word holds 32 imaginary-time sites of ONE
// system: with M = L_tau / 32, site (x, y, tau) is bit tau / M of word-site
// x + L y + L^2 (tau mod M).  M is even, so all bits of a word have the
// colour (x + y + tau) mod 2 of their word-site, and the six neighbours of a
// word are whole words: four spatial ones at the same tau, and the words at
// tau +- 1, rotated by one bit where the word stream wraps (tau mod M = M-1
// upwards, 0 downwards), with the antiperiodic sign on the bit that crosses
// tau = L_tau - 1 -> 0.
//
// The update of a word: u = number of unsatisfied bonds of each bit (6 bond
// masks, a bit-sliced 6-input counter), d = the bit's daemon level, and the
// bit flips iff u + d >= 3 (a flip costs 4k(3 - u); P(d >= n) = e^{-4kn}).
// d >= n is "the first n of the daemon words b4, b8, b12 have the bit set",
// so the flip mask is
//   f = [u >= 3] | b4 & ([u = 2] | b8 & ([u = 1] | b12 & [u = 0])).
// Each daemon word comes from one Philox4x32-10 call (the upper halves of
// four 64-bit "50/50" words) and one xoroshiro128++ state step of the same
// 128 bits (the lower halves); byte i of the word is n* of 64-bit word i,
// the bin of the word in the cumulative table of the walker's slot.
//
// What bounds it: integer issue (three Philox calls and twelve look-ups per
// word), so
//   * n* is found from an index of the top kDaemonLutBits bits, staged in
//     shared memory: the words with a given prefix fall in the bins [n_min,
//     n_min + span], so n* = n_min + #{q in [n_min, n_min + span):
//     cumulative(q) <= word}.  An entry is one 32-bit word: the cut point's
//     upper half below the prefix in its top bits (all ones without a cut), a
//     flag for span >= 2, and n_min.  With span <= 1 the byte is n_min plus
//     one comparison of the word's bits below the prefix with the entry as
//     it stands.  A flagged entry holds the number of the cell's row in a
//     second index by the next kDaemonSubBits bits, of entries of the same
//     form.  Only an entry flagged there too, or bits equal to the cut
//     point's (then the lower halves matter), sends the daemon word to the
//     exact path, which computes the xoroshiro step;
//   * the first two Philox rounds of a word's three calls share their products
//     with the site alone, and those with the system are the block's;
//   * a thread walks up the tau' of one column (x, y), two planes a step, so
//     the couplings and neighbour offsets are fixed, and the word above is
//     the next step's word below;
//   * the comparison adds its byte's one by a predicated multiply-add and the
//     round keys are parameters: the logic pipe (62% busy) binds the kernel.
// 423 instructions per word of 32 updates (555 with 8-byte entries, a branch
// per look-up, whole Philox calls and index arithmetic per word): 10 sweeps at
// L = 16, L_tau = 8192, 16 samples 14.25 -> 10.7 ms (11.2 without the last point).
//
// Device arrays (systems walker-major; PT exchanges slot labels only):
//   spins  u32 [a][r][w][L^2 M]       bit = 1 <=> spin -1
//   J      uint8 [a][x + L*y]          bit0: J(+x) = -1, bit1: J(+y) = -1
//   U      u64 [a][r][w][2]            unsatisfied spatial / tau bonds of walker w
//   cum    u64 [n_slots][256]          cumulative(0..254) of Sec. 2.1.1; [255] = 2^64-1
//   lut    u32 [n_slots][kDaemonLutWords]   cut bits | span >= 2 << 8 | n_min by prefix, then the
//                                      second index's rows of 2^kDaemonSubBits
#include <algorithm>
#include <cmath>
#include <cstring>

#include "qisg_internal.cuh"

namespace qisg {
namespace {

constexpr int kBlock = 256;

constexpr uint32_t kSpanFlag = 0x100u;   // index entry: two or more cut points
static_assert((kDaemonLutWords / 4) % kBlock == 0, "the block stages whole 16-byte words");

struct SitesArgs {
  uint32_t *spins;
  const uint8_t *J;
  const int32_t *walker;
  const unsigned long long *cum;
  const uint32_t *lut;
  unsigned long long *U;
  const unsigned long long *d_t;
  unsigned long long *t_copy;  // blue pass: copy t here for the PT pass that advances it (or null)
  uint2 key;
  PhiloxKeys rk;               // its round keys
  FastDiv plane_div, L_div, bps_div, ns_div, nr_div;
  int L, M, plane, n_words;
  int n_slots, n_rep;
  int n_seg, walk;             // segments per column and words of the colour in one (at most)
  int tau_ap;
  uint32_t one;                // 1 as a runtime value (add_if_less)
};

// xoroshiro128++ state step (Blackman and Vigna, 2019) on the 128 bits of a
// Philox output, state (x | y << 32, z | w << 32); returns the new state's
// four 32-bit quarters in the same order.
__device__ __forceinline__ uint4 xoroshiro_step(uint4 x) {
  const unsigned long long s0 = (unsigned long long)x.x | ((unsigned long long)x.y << 32);
  const unsigned long long s1 = (unsigned long long)x.z | ((unsigned long long)x.w << 32);
  const unsigned long long tt = s1 ^ s0;
  const unsigned long long n0 = ((s0 << 49) | (s0 >> 15)) ^ tt ^ (tt << 21);
  const unsigned long long n1 = (tt << 28) | (tt >> 36);
  return make_uint4((uint32_t)n0, (uint32_t)(n0 >> 32), (uint32_t)n1, (uint32_t)(n1 >> 32));
}

// The exact bytes of a daemon word from its Philox output x: lower halves
// from the xoroshiro step, then for every byte the count of the cut points at
// or below the word among its prefix's candidates.  A candidate run ends at
// the first cut point above the word (the cut points do not decrease).
static __device__ __noinline__ uint32_t daemon_exact(uint4 x, const uint32_t *lut, const unsigned long long *cum) {
  const uint4 lo = xoroshiro_step(x);
  uint32_t b = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t hi = pick4(x, i);
    const unsigned long long R = ((unsigned long long)hi << 32) | pick4(lo, i);
    uint32_t n = lut[hi >> (32 - kDaemonLutBits)] & 0xFFu;
    while (n < 255u && cum[n] <= R) ++n;
    b |= n << (8 * i);
  }
  return b;
}

// One daemon word: byte i is n* of the 64-bit word whose upper half is Philox
// output i.  c: the Philox state after two rounds; k: the round keys.
__device__ __forceinline__ uint32_t daemon_word(uint4 c, const PhiloxKeys &k, const uint32_t *lut,
                                                const unsigned long long *cum, uint32_t one) {
#pragma unroll
  for (int i = 2; i < 10; ++i) {   // one wide product per half round: measured faster here than two halves
    const unsigned long long p0 = (unsigned long long)kPhiloxM0 * c.x;
    const unsigned long long p1 = (unsigned long long)kPhiloxM1 * c.z;
    c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ k.k[i].x, (uint32_t)p1, (uint32_t)(p0 >> 32) ^ c.w ^ k.k[i].y,
                   (uint32_t)p0);
  }
  uint32_t e0 = lut[c.x >> (32 - kDaemonLutBits)], e1 = lut[c.y >> (32 - kDaemonLutBits)];
  uint32_t e2 = lut[c.z >> (32 - kDaemonLutBits)], e3 = lut[c.w >> (32 - kDaemonLutBits)];
  const uint32_t x0 = c.x << kDaemonLutBits, x1 = c.y << kDaemonLutBits;
  const uint32_t x2 = c.z << kDaemonLutBits, x3 = c.w << kDaemonLutBits;
  if ((e0 | e1 | e2 | e3) & kSpanFlag) {   // cells with two or more cut points: by the next bits
    auto finer = [&](uint32_t e, uint32_t x) {
      return e & kSpanFlag ? lut[(1 << kDaemonLutBits) + ((e >> kDaemonLutBits) << kDaemonSubBits) + (x >> (32 - kDaemonSubBits))] : e;
    };
    e0 = finer(e0, x0);
    e1 = finer(e1, x1);
    e2 = finer(e2, x2);
    e3 = finer(e3, x3);
  }
  // n_min of the four bytes, plus one where the word's bits exceed the cut's
  // (the entry's low bits do not reach the next cut value: x > e iff the
  // fields compare so)
  uint32_t b = __byte_perm(__byte_perm(e0, e1, 0x0040), __byte_perm(e2, e3, 0x0040), 0x5410);
  add_if_less(b, e0, x0, 1u, one);
  add_if_less(b, e1, x1, 1u << 8, one);
  add_if_less(b, e2, x2, 1u << 16, one);
  add_if_less(b, e3, x3, 1u << 24, one);
  const uint32_t tie = min(min(x0 ^ e0, x1 ^ e1), min(x2 ^ e2, x3 ^ e3));   // < 2^bits: equal fields
  if ((tie >> kDaemonLutBits) == 0u || ((e0 | e1 | e2 | e3) & kSpanFlag)) b = daemon_exact(c, lut, cum);
  return b;
}

__device__ __forceinline__ uint32_t maj3(uint32_t a, uint32_t b, uint32_t c) { return (a & b) | (c & (a | b)); }

// One half sweep (colour 0 = red, 1 = blue).  Block x serves system
// x / blocks_per_sys (sys = (a n_rep + r) n_slots + w) and 256 consecutive
// (segment, column) pairs of it; a thread walks the colour's words of one
// column in one segment along tau'.  The blue pass counts, per system, the
// unsatisfied bonds of its words after the update: every bond has exactly
// one blue end, so this is each bond once.  Chunk 0 of the red pass clears
// the system's counters.  count_only: no update (energies of the stored
// state).
template <bool BLUE>
__global__ void __launch_bounds__(kBlock) sites_half_sweep_kernel(const SitesArgs p, int count_only) {
  __shared__ unsigned long long cum_s[256];
  extern __shared__ __align__(16) uint32_t lut_s[];   // [kDaemonLutWords]
  __shared__ uint32_t red_s[2][kBlock / 32];
  pdl_begin();
  if (BLUE && p.t_copy && blockIdx.x == 0 && threadIdx.x == 0) *p.t_copy = *p.d_t;
  const uint32_t sys = p.bps_div.div(blockIdx.x), chunk = blockIdx.x - sys * p.bps_div.d;
  const uint32_t ar = p.ns_div.div(sys), w = sys - ar * (uint32_t)p.n_slots;   // ar = a * n_rep + r
  const uint32_t a = p.nr_div.div(ar), r = ar - a * (uint32_t)p.n_rep;
  const uint32_t colour = BLUE ? 1u : 0u;
  if (!BLUE && chunk == 0 && threadIdx.x < 2) p.U[(size_t)sys * 2 + threadIdx.x] = 0;
  if (!BLUE && count_only) return;
  // slot of walker w: lane l of every warp reads walker_at[a][r][l] (a plain
  // load: the PT pass before this kernel writes the labels)
  const int lane = threadIdx.x & 31;
  const int32_t wl = lane < p.n_slots ? p.walker[(size_t)ar * p.n_slots + lane] : -1;
  const int s = max(__ffs(__ballot_sync(0xFFFFFFFFu, wl == (int32_t)w)) - 1, 0);   // rows are permutations
  // stage the slot's tables
  if (!count_only) {
    cum_s[threadIdx.x] = __ldg(p.cum + (size_t)s * 256 + threadIdx.x);
    const uint4 *lg = reinterpret_cast<const uint4 *>(p.lut + (size_t)s * kDaemonLutWords);
    uint4 *ls = reinterpret_cast<uint4 *>(lut_s);
#pragma unroll
    for (int i = 0; i < kDaemonLutWords / 4 / kBlock; ++i) ls[i * kBlock + threadIdx.x] = __ldg(lg + i * kBlock + threadIdx.x);
    __syncthreads();
  }
  const uint32_t P = (uint32_t)p.plane, L = (uint32_t)p.L, M = (uint32_t)p.M;
  const uint32_t gq = chunk * (uint32_t)kBlock + threadIdx.x;   // (segment, column)
  const uint32_t seg = p.plane_div.div(gq), i2 = gq - seg * P;
  uint32_t us_cnt = 0, ut_cnt = 0;
  if (seg < (uint32_t)p.n_seg) {
    const uint32_t y = p.L_div.div(i2), x = i2 - y * L;
    const uint32_t ixp = x + 1 == L ? i2 + 1 - L : i2 + 1, ixm = x == 0 ? i2 + L - 1 : i2 - 1;
    const uint32_t iyp = y + 1 == L ? x : i2 + L, iym = y == 0 ? i2 + P - L : i2 - L;
    const uint8_t *J = p.J + (size_t)a * P;
    const uint32_t jc = __ldg(J + i2);
    const uint32_t Jxp = 0u - (jc & 1u), Jxm = 0u - (__ldg(J + ixm) & 1u);
    const uint32_t Jyp = 0u - ((jc >> 1) & 1u), Jym = 0u - ((__ldg(J + iym) >> 1) & 1u);
    uint32_t *S = p.spins + (size_t)sys * p.n_words;
    const uint32_t t = (uint32_t)*p.d_t;
    const uint32_t c3 = (DOM_DAEMON << 28) | a;
    // Philox rounds 1 and 2, the products of the system's counter word
    const uint32_t c2 = (uint32_t)s | (r << 16);
    const uint32_t y1 = kPhiloxM1 * c2 ^ (p.key.x + kPhiloxW0), h1 = __umulhi(kPhiloxM1, c2) ^ t ^ p.key.x;
    const uint32_t X = __umulhi(kPhiloxM0, h1) ^ (p.key.y + kPhiloxW1), w2 = kPhiloxM0 * h1;
    const uint32_t ap_up = p.tau_ap ? 0x80000000u : 0u, ap_dn = p.tau_ap ? 1u : 0u;
    uint32_t tq = ((x + y + colour) & 1u) + 2u * seg * (uint32_t)p.walk;
    const uint32_t end = min(M, 2u * (seg + 1) * (uint32_t)p.walk);
    uint32_t dn = 0;
    if (tq < end) {
      dn = S[i2 + P * (tq == 0 ? M - 1 : tq - 1)];
      if (tq == 0) dn = __funnelshift_l(dn, dn, 1) ^ ap_dn;   // bit j <- bit j-1 of tau' = M-1
    }
    for (; tq < end; tq += 2) {
      const uint32_t off = P * tq, ws = i2 + off;
      const bool top = tq + 1 == M;
      const uint32_t c = S[ws], sxp = S[ixp + off], sxm = S[ixm + off], syp = S[iyp + off], sym = S[iym + off];
      const uint32_t above = S[top ? i2 : ws + P];
      uint32_t b4 = 0, b8 = 0, b12 = 0;
      if (!count_only) {
        // rounds 1 and 2, the products of the word-site; the three words
        // differ in the last counter word
        const uint32_t zs = __umulhi(kPhiloxM0, ws) ^ p.key.y ^ c3, z2 = (kPhiloxM0 * ws) ^ X;
        // b4, b8, b12 in a rolled loop (one copy of the look-up code)
#pragma unroll 1
        for (uint32_t which = 0; which < 3; ++which) {
          const uint32_t z1 = zs ^ (which << 24);
          const uint32_t dw =
              daemon_word(make_uint4(__umulhi(kPhiloxM1, z1) ^ y1, kPhiloxM1 * z1, z2, w2), p.rk, lut_s, cum_s, p.one);
          b4 = b8;
          b8 = b12;
          b12 = dw;
        }
      }
      const uint32_t up = top ? __funnelshift_r(above, above, 1) ^ ap_up : above;   // bit j <- bit j+1 of tau' = 0
      // unsatisfied bond masks: J S S' = -1 <=> bit(S) ^ bit(S') ^ bit(J) = 1
      const uint32_t e1 = c ^ sxp ^ Jxp, e2 = c ^ sxm ^ Jxm, e3 = c ^ syp ^ Jyp, e4 = c ^ sym ^ Jym;
      const uint32_t e5 = c ^ up, e6 = c ^ dn;
      uint32_t f = 0;
      if (!count_only) {
        // u = u0 + 2 u1 + 4 u2, bit-sliced over the 32 sites
        const uint32_t s1 = e1 ^ e2 ^ e3, k1 = maj3(e1, e2, e3);
        const uint32_t s2 = e4 ^ e5 ^ e6, k2 = maj3(e4, e5, e6);
        const uint32_t u0 = s1 ^ s2, h = s1 & s2;
        const uint32_t u1 = k1 ^ k2 ^ h, u2 = maj3(k1, k2, h);
        const uint32_t ge3 = u2 | (u1 & u0);
        const uint32_t eq2 = ~u2 & u1 & ~u0, eq1 = ~u2 & ~u1 & u0, eq0 = ~(u2 | u1 | u0);
        f = ge3 | (b4 & (eq2 | (b8 & (eq1 | (b12 & eq0)))));
        S[ws] = c ^ f;
      }
      if (BLUE) {
        us_cnt += __popc(e1 ^ f) + __popc(e2 ^ f) + __popc(e3 ^ f) + __popc(e4 ^ f);
        ut_cnt += __popc(e5 ^ f) + __popc(e6 ^ f);
      }
      dn = above;   // the next word of the walk is two planes up
    }
  }
  if (BLUE) {   // at most 2^7 x walk per thread, walk <= 2^14: 32 bits hold the block's sum
    us_cnt = __reduce_add_sync(0xFFFFFFFFu, us_cnt);
    ut_cnt = __reduce_add_sync(0xFFFFFFFFu, ut_cnt);
    if (lane == 0) {
      red_s[0][threadIdx.x >> 5] = us_cnt;
      red_s[1][threadIdx.x >> 5] = ut_cnt;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
      unsigned long long v = 0;
      for (int i = 0; i < kBlock / 32; ++i) v += red_s[threadIdx.x][i];
      if (v) atomicAdd(p.U + (size_t)sys * 2 + threadIdx.x, v);
    }
  }
}

// Overlaps of the configurations at slot s (Appendix E.1): count the sites
// where the replicas r1 < r2 differ (popcount of the XOR of their words);
// q = N - 2 * count.  Grid (chunks, n_slots, n_a).
__global__ void __launch_bounds__(kBlock) sites_overlap_kernel(const uint32_t *spins, const int32_t *walker,
                                                               long long *qcnt, int64_t a0, int n_words,
                                                               int n_rep, int n_slots) {
  extern __shared__ long long q_s[];  // [n_pairs]
  const int n_pairs = n_rep * (n_rep - 1) / 2;
  const int s = blockIdx.y;
  const int64_t a = a0 + blockIdx.z;
  for (int i = threadIdx.x; i < n_pairs; i += blockDim.x) q_s[i] = 0;
  __syncthreads();
  const int32_t *wa = walker + a * n_rep * n_slots;
  int p = 0;
  for (int r1 = 0; r1 < n_rep; ++r1) {
    const uint32_t *S1 = spins + ((a * n_rep + r1) * n_slots + wa[r1 * n_slots + s]) * (int64_t)n_words;
    for (int r2 = r1 + 1; r2 < n_rep; ++r2, ++p) {
      const uint32_t *S2 = spins + ((a * n_rep + r2) * n_slots + wa[r2 * n_slots + s]) * (int64_t)n_words;
      unsigned cnt = 0;
      for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_words; i += gridDim.x * blockDim.x)
        cnt += __popc(S1[i] ^ S2[i]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xFFFFFFFFu, cnt, o);
      if ((threadIdx.x & 31) == 0 && cnt)
        atomicAdd(reinterpret_cast<unsigned long long *>(&q_s[p]), (unsigned long long)cnt);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n_pairs; i += blockDim.x)
    if (q_s[i])
      atomicAdd(reinterpret_cast<unsigned long long *>(&qcnt[(a * n_slots + s) * n_pairs + i]),
                (unsigned long long)q_s[i]);
}

// Start spins from Philox domain DOM_INIT: one thread per word, 32 draws.
__global__ void sites_init_spins_kernel(uint32_t *spins, int64_t n_sys, int n_words, int L, int M, int n_rep,
                                        int n_slots, uint2 key) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= n_sys * n_words) return;
  const int ws = (int)(c % n_words);
  const int64_t sys = c / n_words;
  const int w = (int)(sys % n_slots);
  const int64_t ar = sys / n_slots;
  const int r = (int)(ar % n_rep);
  const int64_t a = ar / n_rep;
  const int plane = L * L;
  const int tq = ws / plane, i2 = ws - tq * plane;
  uint32_t v = 0;
  for (int j = 0; j < 32; ++j) {
    const uint32_t site = (uint32_t)(i2 + plane * (tq + j * M));
    const uint4 x = philox(make_uint4(site, (uint32_t)w, (uint32_t)a, (DOM_INIT << 28) | (uint32_t)r), key);
    if (!(x.x & 1u)) v |= 1u << j;   // spin -1
  }
  spins[c] = v;
}

// int8 +-1 spins [sys][site] of systems sys0 .. sys0+n_sys-1 from the
// lattice (site (x, y, tau) is bit tau / M of word x + L y + L^2 (tau mod M)).
__global__ void sites_extract_kernel(const uint32_t *spins, int8_t *out, int64_t sys0, int64_t n_sys, int plane,
                                     int M, int n_words, int64_t N) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= n_sys * N) return;
  const int64_t sys = c / N, site = c - sys * N;
  const int tau = (int)(site / plane), i2 = (int)(site - (int64_t)tau * plane);
  const uint32_t v = spins[(sys0 + sys) * n_words + i2 + plane * (tau % M)];
  out[c] = ((v >> (tau / M)) & 1u) ? -1 : 1;
}

// The words of systems sys0 .. sys0+n_sys-1 from int8 +-1 spins staged as
// [sys][site]: a thread per word, 32 spins along tau.
__global__ void sites_pack_kernel(uint32_t *spins, const int8_t *stage, int64_t sys0, int64_t n_sys, int plane, int M,
                                  int n_words, int64_t N) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= n_sys * n_words) return;
  const int64_t sys = c / n_words;
  const int ws = (int)(c - sys * n_words), tq = ws / plane, i2 = ws - tq * plane;
  uint32_t v = 0;
  for (int j = 0; j < 32; ++j)
    if (stage[sys * N + i2 + (int64_t)plane * (tq + j * M)] == -1) v |= 1u << j;
  spins[(sys0 + sys) * n_words + ws] = v;
}

SitesArgs make_args(qisg_handle *h) {
  SitesArgs p;
  p.spins = reinterpret_cast<uint32_t *>(h->spins);
  p.J = reinterpret_cast<const uint8_t *>(h->J);
  p.walker = h->d_walker;
  p.cum = h->d_dcum;
  p.lut = h->d_dlut;
  p.U = h->d_U;
  p.d_t = h->d_t;
  p.t_copy = nullptr;
  p.key = make_uint2((uint32_t)h->seed, (uint32_t)(h->seed >> 32));
  p.rk = PhiloxKeys(p.key);
  p.L = h->L;
  p.M = h->Lt / 32;
  p.plane = h->L * h->L;
  p.n_words = p.plane * p.M;
  p.plane_div = FastDiv((uint32_t)p.plane);
  p.L_div = FastDiv((uint32_t)h->L);
  p.n_slots = h->n_slots;
  p.n_rep = h->n_rep;
  p.ns_div = FastDiv((uint32_t)h->n_slots);
  p.nr_div = FastDiv((uint32_t)h->n_rep);
  p.tau_ap = h->tau_ap;
  p.one = 1u;
  // words per walk: up to 16 (a block stages 40 KB of tables for its 256
  // walks; ms per sweep at 8 | 16 | 32 words: L = 16, L_tau = 8192 1.119 | 1.100
  // | 1.096, L = 24, L_tau = 2048 0.641 | 0.643 | 0.701) while the grid keeps 8
  // blocks per SM
  const int64_t n_sys = h->n_samples * h->n_rep * h->n_slots;
  const int half = p.M / 2;
  int walk = std::min(half, h->sweep_tile[0] > 0 ? h->sweep_tile[0] : 16);
  auto per_sys = [&](int g) { return ((int64_t)p.plane * ((half + g - 1) / g) + kBlock - 1) / kBlock; };
  while (walk > 1 && n_sys * per_sys(walk) < 8LL * h->n_sm) walk >>= 1;
  p.walk = walk;
  p.n_seg = (half + walk - 1) / walk;
  p.bps_div = FastDiv((uint32_t)per_sys(walk));
  return p;
}

// Fixed-point numbers in [0, 2) with 126 fractional bits.
using u128 = unsigned __int128;
constexpr int kFrac = 126;
const u128 kOne = (u128)1 << kFrac;

// floor(a b / 2^126) for a, b < 2^127, through 64-bit limbs.
u128 mulq(u128 a, u128 b) {
  const uint64_t a0 = (uint64_t)a, a1 = (uint64_t)(a >> 64), b0 = (uint64_t)b, b1 = (uint64_t)(b >> 64);
  const u128 p00 = (u128)a0 * b0, p01 = (u128)a0 * b1, p10 = (u128)a1 * b0, p11 = (u128)a1 * b1;
  const u128 mid = (p00 >> 64) + (uint64_t)p01 + (uint64_t)p10;
  const u128 hi = p11 + (p01 >> 64) + (p10 >> 64) + (mid >> 64);   // bits 128..255
  const u128 lo = (mid << 64) | (uint64_t)p00;                       // bits 0..127
  return (hi << (128 - kFrac)) | (lo >> kFrac);
}

// e^{-x} for 0 <= x <= 64 in fixed point: x = y 2^m with y < 1/16 (exact),
// e^{-y} by its Taylor series (terms to y^30/30!), then m squarings.
u128 exp_neg(double x) {
  int m = 0;
  while (x / std::ldexp(1.0, m) >= 1.0 / 16) ++m;
  const double y = x / std::ldexp(1.0, m);   // exact: a power-of-two scaling
  int ex = 0;
  const double fr = std::frexp(y, &ex);     // y = fr 2^ex, fr in [0.5, 1)
  const uint64_t mant = (uint64_t)std::ldexp(fr, 53);
  const int sh = kFrac + ex - 53;
  const u128 yq = y == 0.0 ? 0 : (sh >= 0 ? (u128)mant << sh : (u128)(mant >> (-sh)));
  u128 term = kOne, pos = kOne, neg = 0;
  for (int i = 1; i <= 30; ++i) {
    term = mulq(term, yq) / (u128)i;
    if (i & 1) neg += term;
    else pos += term;
  }
  u128 r = pos - neg;
  for (int i = 0; i < m; ++i) r = mulq(r, r);
  return r;
}

}  // namespace

// cumulative(0..254) of Sec. 2.1.1 for coupling k (0 <= k <= 16):
// floor(2^64 sum_{m <= n} p^pop(m) (1-p)^(8-pop(m))), p = e^{-4k}, in
// fixed point with 126 fractional bits (the paper uses 128-bit floats).
void daemon_cumulative(double k, uint64_t *cum) {
  const u128 p = exp_neg(4.0 * k);
  const u128 q = kOne - p;
  u128 pw[9], qw[9];
  pw[0] = qw[0] = kOne;
  for (int c = 1; c <= 8; ++c) {
    pw[c] = mulq(pw[c - 1], p);
    qw[c] = mulq(qw[c - 1], q);
  }
  u128 acc = 0;
  for (int n = 0; n < 255; ++n) {
    const int c = __builtin_popcount((unsigned)n);
    acc += mulq(pw[c], qw[8 - c]);
    cum[n] = (uint64_t)(acc >> (kFrac - 64));
  }
}

// Prefix index of one cumulative table: entry h covers the words
// [h 2^(64-bits), (h+1) 2^(64-bits)), whose n* lie in [n_min, n_max];
// entry = n_min | (n_max - n_min) << 8.
void daemon_lut(const uint64_t *cum, int bits, uint16_t *lut) {
  auto ns = [&](uint64_t R) {
    uint32_t c = 0;
    while (c < 255 && cum[c] <= R) ++c;   // cum is non-decreasing
    return c;
  };
  for (uint64_t h = 0; h < (1ull << bits); ++h) {
    const uint64_t lo = h << (64 - bits), hi = lo + ((~0ull) >> bits);
    const uint32_t a = ns(lo), b = ns(hi);
    lut[h] = (uint16_t)(a | ((b - a) << 8));
  }
}

int sites_build_tables(qisg_handle *h) {
  const int n = h->n_slots;
  std::vector<unsigned long long> cum((size_t)n * 256);
  std::vector<uint32_t> lut((size_t)n * kDaemonLutWords, 0u);
  for (int s = 0; s < n; ++s) {
    uint64_t c[256];
    daemon_cumulative(h->k[s], c);
    c[255] = ~0ull;
    for (int i = 0; i < 256; ++i) cum[(size_t)s * 256 + i] = c[i];
    auto nstar = [&](uint64_t R) { return (uint32_t)(std::upper_bound(c, c + 255, R) - c); };
    // entry of the words with the top `bits` bits h: *span gets the number of
    // cut points inside the cell
    auto entry = [&](uint64_t h, int bits, uint32_t *span) {
      const uint64_t lo = h << (64 - bits);
      const uint32_t nmin = nstar(lo);
      *span = nstar(lo + ((~0ull) >> bits)) - nmin;
      // the one cut point's upper half below the prefix, else all ones
      const uint32_t cut = *span == 1 ? (uint32_t)(c[nmin] >> 32) << kDaemonLutBits : 0xFFFFFFFFu << kDaemonLutBits;
      return cut | (*span >= 2 ? kSpanFlag : 0u) | nmin;
    };
    uint32_t *out = &lut[(size_t)s * kDaemonLutWords];
    uint32_t row = 0, span;   // cells with two or more of the 255 cut points: at most 127
    for (uint64_t i = 0; i < (1ull << kDaemonLutBits); ++i) {
      out[i] = entry(i, kDaemonLutBits, &span);
      if (span < 2) continue;
      out[i] = (row << kDaemonLutBits) | kSpanFlag | (out[i] & 0xFFu);
      uint32_t *sub = out + (1 << kDaemonLutBits) + (row++ << kDaemonSubBits);
      for (uint64_t j = 0; j < (1ull << kDaemonSubBits); ++j)
        sub[j] = entry((i << kDaemonSubBits) | j, kDaemonLutBits + kDaemonSubBits, &span);
    }
  }
  int rc = cuda_check(cudaMemcpyAsync(h->d_dcum, cum.data(), cum.size() * 8, cudaMemcpyHostToDevice, h->stream),
                      "copy cumulative tables");
  if (!rc)
    rc = cuda_check(cudaMemcpyAsync(h->d_dlut, lut.data(), lut.size() * 4, cudaMemcpyHostToDevice, h->stream),
                    "copy prefix index");
  // the host vectors must outlive the copies
  if (!rc) rc = cuda_check(cudaStreamSynchronize(h->stream), "sync");
  return rc;
}

int sites_init(qisg_handle *h) {
  int rc = sites_build_tables(h);
  if (rc) return rc;
  const uint2 key = make_uint2((uint32_t)h->seed, (uint32_t)(h->seed >> 32));
  rc = lanes_init_couplings(h);
  if (rc) return rc;
  const int n_words = h->L * h->L * (h->Lt / 32);
  const int64_t n_sys = h->n_samples * h->n_rep * h->n_slots;
  const int64_t nS = n_sys * n_words;
  if ((nS + 255) / 256 > 0x7FFFFFFF) return fail(QISG_EINVAL, "lattice too large");
  sites_init_spins_kernel<<<(unsigned)((nS + 255) / 256), 256, 0, h->stream>>>(
      reinterpret_cast<uint32_t *>(h->spins), n_sys, n_words, h->L, h->Lt / 32, h->n_rep, h->n_slots, key);
  h->launches++;
  return cuda_check(cudaGetLastError(), "sites init");
}

int sites_half_sweep(qisg_handle *h, int colour, int count_only) {
  SitesArgs p = make_args(h);
  if (colour == 1 && !count_only && lanes_pt_advances(h)) p.t_copy = h->d_t + 1;
  const int64_t n_sys = h->n_samples * h->n_rep * h->n_slots;
  const int64_t blocks = n_sys * p.bps_div.d;
  if (blocks > 0x7FFFFFFF) return fail(QISG_EINVAL, "lattice too large for one launch");
  constexpr size_t smem = sizeof(uint32_t) * kDaemonLutWords;
  static bool attr_set = false;
  if (!attr_set) {
    cudaFuncSetAttribute(sites_half_sweep_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(sites_half_sweep_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    attr_set = true;
  }
  const int tok = prof_begin(h, sweep_kind(colour));
  launch_kernel(h->pdl, colour == 1 ? sites_half_sweep_kernel<true> : sites_half_sweep_kernel<false>,
                dim3((unsigned)blocks), dim3(kBlock), smem, h->stream, p, count_only);
  prof_end(h, sweep_kind(colour), tok);
  h->launches++;
  return cuda_check(cudaGetLastError(), "sites half sweep");
}

int sites_measure(qisg_handle *h, int force_to_q) {
  const int n_pairs = h->n_pairs();
  if (n_pairs > 0) {
    const int n_words = h->L * h->L * (h->Lt / 32);
    const int64_t chunks = std::min<int64_t>((n_words + kBlock - 1) / kBlock, 64);
    const size_t smem = (size_t)n_pairs * 8;
    for (int64_t a0 = 0; a0 < h->n_samples; a0 += 65535) {
      const int64_t na = std::min<int64_t>(65535, h->n_samples - a0);
      const int tok = prof_begin(h, QISG_KERNEL_MEASURE);
      sites_overlap_kernel<<<dim3((unsigned)chunks, (unsigned)h->n_slots, (unsigned)na), kBlock, smem,
                             h->stream>>>(reinterpret_cast<const uint32_t *>(h->spins), h->d_walker, h->d_q, a0,
                                          n_words, h->n_rep, h->n_slots);
      prof_end(h, QISG_KERNEL_MEASURE, tok);
      h->launches++;
    }
    int rc = cuda_check(cudaGetLastError(), "sites overlaps");
    if (rc) return rc;
  }
  return lanes_finalize(h, force_to_q);
}

int sites_stage_spins(qisg_handle *h, int64_t a_lo, int64_t n_a, int8_t *d) {
  const int M = h->Lt / 32, plane = h->L * h->L, n_words = plane * M;
  const int64_t n_sys = n_a * h->n_rep * h->n_slots, n = n_sys * h->N;
  if (n == 0) return QISG_OK;
  sites_extract_kernel<<<(unsigned)((n + 255) / 256), 256, 0, h->stream>>>(
      reinterpret_cast<const uint32_t *>(h->spins), d, a_lo * h->n_rep * h->n_slots, n_sys, plane, M, n_words, h->N);
  h->launches++;
  return cuda_check(cudaGetLastError(), "unpack spins");
}

int sites_get_spins(qisg_handle *h, int64_t a_lo, int64_t n_a, int8_t *S) {
  const int M = h->Lt / 32, plane = h->L * h->L, n_words = plane * M;
  const int64_t per_sys = h->N, n_sys = n_a * h->n_rep * h->n_slots, sys_lo = a_lo * h->n_rep * h->n_slots;
  if (n_sys == 0) return QISG_OK;
  const int64_t chunk = std::min<int64_t>(n_sys, std::max<int64_t>(1, ((int64_t)256 << 20) / per_sys));
  int8_t *stage = nullptr;
  int rc = cuda_check(cudaMalloc(&stage, (size_t)(chunk * per_sys)), "cudaMalloc");
  for (int64_t s0 = 0; s0 < n_sys && !rc; s0 += chunk) {
    const int64_t ns = std::min(chunk, n_sys - s0), n = ns * per_sys;
    sites_extract_kernel<<<(unsigned)((n + 255) / 256), 256, 0, h->stream>>>(
        reinterpret_cast<const uint32_t *>(h->spins), stage, sys_lo + s0, ns, plane, M, n_words, h->N);
    h->launches++;
    rc = cuda_check(cudaGetLastError(), "unpack spins");
    if (!rc)
      rc = cuda_check(cudaMemcpyAsync(S + s0 * per_sys, stage, (size_t)n, cudaMemcpyDeviceToHost, h->stream), "copy");
    if (!rc) rc = cuda_check(cudaStreamSynchronize(h->stream), "sync");
  }
  if (stage) cudaFree(stage);
  return rc;
}

int sites_set_spins(qisg_handle *h, const int8_t *S) {
  const int M = h->Lt / 32, plane = h->L * h->L, n_words = plane * M;
  const int64_t per_sys = h->N, n_sys = h->n_samples * h->n_rep * h->n_slots;
  const int64_t chunk = std::min<int64_t>(n_sys, std::max<int64_t>(1, ((int64_t)256 << 20) / per_sys));
  int8_t *stage = nullptr;
  int rc = cuda_check(cudaMalloc(&stage, (size_t)(chunk * per_sys)), "cudaMalloc");
  for (int64_t s0 = 0; s0 < n_sys && !rc; s0 += chunk) {
    const int64_t ns = std::min(chunk, n_sys - s0), n = ns * n_words;
    rc = cuda_check(cudaMemcpyAsync(stage, S + s0 * per_sys, (size_t)(ns * per_sys), cudaMemcpyHostToDevice,
                                    h->stream),
                    "copy spins");
    if (rc) break;
    sites_pack_kernel<<<(unsigned)((n + 255) / 256), 256, 0, h->stream>>>(reinterpret_cast<uint32_t *>(h->spins),
                                                                          stage, s0, ns, plane, M, n_words, h->N);
    h->launches++;
    rc = cuda_check(cudaGetLastError(), "pack spins");
  }
  if (!rc) rc = cuda_check(cudaStreamSynchronize(h->stream), "sync");
  if (stage) cudaFree(stage);
  return rc;
}

}  // namespace qisg

extern "C" int qisg_daemon_tables(double k, int lut_bits, uint64_t *cum, uint16_t *lut) {
  if (!cum || !(k >= 0.0) || !(k <= 16.0)) return qisg::fail(QISG_EINVAL, "need 0 <= k <= 16 and a table");
  if (lut && (lut_bits < 1 || lut_bits > 16)) return qisg::fail(QISG_EINVAL, "lut_bits must be in 1..16");
  qisg::daemon_cumulative(k, cum);
  if (lut) qisg::daemon_lut(cum, lut_bits, lut);
  return QISG_OK;
}
