// Half sweep of one sample in the LANES packing.
//
// A 32- or 64-bit word holds replicas x walkers of the sample: lane =
// (r - g*rpw) * n_slots + w in word group g = r / rpw.  The thread of a site
// loads the site's and its six neighbours' words once, forms the bit-sliced
// counts u_s (4 spatial bonds) and u_t (2 tau bonds) of every lane, and then
// visits every (slot s, replica r): the walker w at slot s of replica r is
// lane (r, w), whose draw R (one Philox call per (slot, replica quad, site,
// sweep)) is compared with the threshold T[s][u_s][u_t] (Sec. 2.1).
//
// What bounds it: integer issue, one Philox call per four updates and the
// look-up of each lane's threshold.  So
//   * the classes that always flip (u_t >= 1, u_s >= 2) share codes, which
//     leaves a 4-bit class code; the four code planes become a byte per lane
//     (code * 4, the byte offset in a 16-entry threshold row) by a 4 x 4
//     nibble transposition, one operation per lane, kept in shared memory;
//   * lane offsets and flip bits of each (slot, replica) are uniform over the
//     block and come from a small table, so an update is: code byte, its
//     threshold, compare, set a bit of the replica's 32-bit flip mask;
//   * the first two Philox rounds separate: with the counter (site, t, s | q
//     << 16, w) their products depend on the site alone or on (s, q) alone,
//     so a call costs eight rounds and two exclusive-ors.
// 22.8 thread instructions per update on the uneven batch, 54 with a byte
// spread of five planes, plane tables in shared memory and whole Philox calls:
// 20 sweeps of 512 instances took 265.6 ms, then 155.4.
//
// In the blue pass the unsatisfied bonds after the flip are accumulated per
// lane in bit-sliced counters; after at most seven sites per thread each
// plane is transposed across the warp (32 x 32 bits, five shuffles), so a
// lane's sum over the warp is one popcount per plane (every bond has exactly
// one blue end).
//
// TPS = 1: a thread per site.  TPS = 4: four warps share 32 sites, each
// taking every fourth slot (and one 32-bit half of the words), for launches
// with too few sites to fill the GPU.
#pragma once

#include "qisg_internal.cuh"

namespace qisg {

constexpr int kLanesMaxGroups = 2;    // word groups per site held in registers
constexpr int kLanesMaxRows = 16;     // rows of kLanesThreads sites in a tile (a choice: the counters are flushed every seven)
constexpr int kLanesKs = 5;           // u_s counter planes: <= 4 x 7 sites per thread
constexpr int kLanesKt = 4;           // u_t counter planes: <= 2 x 7 sites per thread
constexpr int kLanesFlushSites = 7;   // sites per thread between flushes of the counters
constexpr int kLanesThreads = 256;                       // block size
constexpr int kLanesCodeWords = kLanesMaxGroups * 16;    // per site: 2 groups x 64 lanes, 4 per word

template <typename Word>
struct LanesSample {
  Word *spins;                   // [g][N]
  const uint32_t *T;             // [n_slots][15] (global)
  const int32_t *walker;         // [r][s]
  unsigned long long *U;         // [r][w][2], by walker
  const uint8_t *J;              // [L*L]
  uint2 key;
  uint32_t ctr_w;                // (DOM_SWEEP << 28) | (a >> 6)
  uint32_t t;                    // sweep index
  FastDiv hpd, hld;              // by plane / 2 and by L / 2
  uint32_t N;                    // sites (up to 2^31)
  int L, Lt, plane, half_plane, n_slots, n_rep, rpw, n_groups;
  uint32_t one;                  // 1 as a runtime value (add_if_less)
  int tau_ap;                    // antiperiodic along tau: the wrap tau bond flips sign
};

// Shared memory of one tile: threshold rows by class code, the lane table,
// the Philox words of each (slot, quad), counter sums, the flips that the
// TPS = 4 form exchanges, and the class codes.  At most 41472 bytes (32 slots x
// 4 replicas), so no kernel that runs tiles has to raise the 48 KB that a launch
// may ask for.
__host__ __device__ inline size_t lanes_tile_smem(int n_slots, int n_rep) {
  const size_t sq = (size_t)n_slots * ((n_rep + 3) / 4);
  size_t o = sq * 48 + (size_t)n_slots * 64;                  // lane table and Philox words, threshold rows
  o += (size_t)2 * kLanesMaxGroups * 64 * 4;                  // acc_s, acc_t
  o += (size_t)2 * kLanesMaxGroups * kLanesThreads * 4;       // fx
  o += (size_t)kLanesCodeWords * kLanesThreads * 4;
  return (o + 15) & ~size_t(15);
}

template <bool CG, typename Word>
__device__ __forceinline__ Word ld_word(const Word *p) {
  return CG ? __ldcg(p) : *p;
}

// Class code planes of 32 lanes: code = u_s at u_t = 0, else 8 + (u_s & 1) +
// 2 [u_t = 2] + 4 [u_s >= 2] (those with bit 2 set always flip).  The codes
// times 4 go to eight words, a byte per lane: lane l is byte l >> 3 of word
// 2 (l & 3) + ((l >> 2) & 1) (kLanesThreads words apart).
__device__ __forceinline__ void lanes_store_codes(uint32_t *cw, uint32_t P0, uint32_t P1, uint32_t P2, uint32_t Q0,
                                                  uint32_t Q1) {
  const uint32_t nz = Q0 | Q1;
  const uint32_t c1 = mux(nz, Q1, P1), c2 = P2 | (nz & P1);
  // 4 x 4 transposition of the planes' nibbles: bit i of nibble k of word j
  // becomes bit j of nibble k of plane i
  const uint32_t a0 = mux(0x55555555u, P0, c1 << 1), a1 = mux(0x55555555u, P0 >> 1, c1);
  const uint32_t a2 = mux(0x55555555u, c2, nz << 1), a3 = mux(0x55555555u, c2 >> 1, nz);
  const uint32_t w[4] = {mux(0x33333333u, a0, a2 << 2), mux(0x33333333u, a1, a3 << 2),
                         mux(0x33333333u, a0 >> 2, a2), mux(0x33333333u, a1 >> 2, a3)};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    cw[(2 * j) * kLanesThreads] = (w[j] << 2) & 0x3C3C3C3Cu;
    cw[(2 * j + 1) * kLanesThreads] = (w[j] >> 2) & 0x3C3C3C3Cu;
  }
}

// Sites [j0, j0 + n) of one colour; every thread of the block must call it
// (kLanesThreads threads).  NREP > 0: the sample has exactly NREP <= 4
// replicas (one quad).  NGC > 0: exactly NGC word groups per site (registers
// for those only).
// CG: read mutable state through L2 only (inside a persistent kernel).
// zero_U: clear this sample's bond counters first (red pass, one tile).
template <typename Word, bool CG, bool BLUE, int NREP = 0, int NGC = 0, int TPS = 1>
__device__ void lanes_tile(const LanesSample<Word> &S, int colour, int j0, int n, int count_only, bool zero_U,
                           unsigned char *smem) {
  constexpr int W = (int)sizeof(Word) * 8, HW = W / 32;
  constexpr int MG = NGC > 0 ? NGC : kLanesMaxGroups;   // word groups held in registers
  constexpr int MH = MG * HW;                             // 32-bit halves of them
  constexpr int NH = TPS == 1 ? MH : (MH + TPS - 1) / TPS;   // halves of this thread
  constexpr int SPI = kLanesThreads / TPS;                // sites per iteration of the block
  static_assert(SPI % 32 == 0, "a warp's threads share their part of the slots");
  const int n_slots = S.n_slots, n_rep = NREP > 0 ? NREP : S.n_rep, plane = S.plane, hp = S.half_plane;
  const int nq = NREP > 0 ? 1 : (n_rep + 3) >> 2, sq = n_slots * nq;
  const int NG = NGC > 0 ? NGC : S.n_groups;             // 1 or 2
  uint4 *inf = reinterpret_cast<uint4 *>(smem);          // [s][q][2]: {code offset, flip bit} of four replicas
  uint4 *phx = inf + 2 * sq;                               // [s][q]: the (s, q) words of Philox rounds 1 and 2
  uint32_t *T16 = reinterpret_cast<uint32_t *>(phx + sq);   // [slot][code]
  int *acc_s = reinterpret_cast<int *>(T16 + n_slots * 16);   // [group][lane]
  int *acc_t = acc_s + kLanesMaxGroups * 64;
  uint32_t *fx = reinterpret_cast<uint32_t *>(acc_t + kLanesMaxGroups * 64);   // [half][part][site]
  uint32_t *code_s = fx + 2 * kLanesMaxGroups * kLanesThreads;                 // [word][site]

  __syncthreads();   // a previous tile is done with shared memory
  for (int i = threadIdx.x; i < n_slots * 16; i += kLanesThreads) {
    const int c = i & 15, us = c < 8 ? c : c & 1, ut = c < 8 ? 0 : 1 + ((c >> 1) & 1);
    T16[i] = (c < 8 ? us <= 4 : !(c & 4)) ? S.T[(i >> 4) * 15 + us * 3 + ut] : 0xFFFFFFFFu;
  }
  for (int i = threadIdx.x; i < sq; i += kLanesThreads) {
    const int s = i / nq, q = i - s * nq;
    uint32_t e[8];
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
      const int r = 4 * q + jj;
      uint32_t off = 0, bit = 0;
      if (r < n_rep) {
        const int w = CG ? __ldcg(S.walker + r * n_slots + s) : S.walker[r * n_slots + s];
        const int g = r / S.rpw, l = (r - g * S.rpw) * n_slots + w;   // lane of group g
        off = (uint32_t)((g * 16 + (l >> 5) * 8 + 2 * (l & 3) + ((l >> 2) & 1)) * kLanesThreads * 4 + ((l & 31) >> 3));
        bit = 1u << w;
      }
      e[2 * jj] = off;
      e[2 * jj + 1] = bit;
    }
    inf[2 * i] = make_uint4(e[0], e[1], e[2], e[3]);
    inf[2 * i + 1] = make_uint4(e[4], e[5], e[6], e[7]);
    const uint32_t cz = (uint32_t)s | ((uint32_t)q << 16);
    const uint32_t x1 = __umulhi(kPhiloxM1, cz) ^ S.t ^ S.key.x;
    phx[i] = make_uint4(kPhiloxM1 * cz, __umulhi(kPhiloxM0, x1), kPhiloxM0 * x1, 0u);
  }
  if (BLUE)
    for (int i = threadIdx.x; i < 2 * kLanesMaxGroups * 64; i += kLanesThreads) acc_s[i] = 0;
  if (zero_U)
    for (int i = threadIdx.x; i < 2 * n_rep * n_slots; i += kLanesThreads) S.U[i] = 0;
  __syncthreads();

  const int sl = TPS == 1 ? (int)threadIdx.x : (int)threadIdx.x % SPI;   // site of the iteration
  const int part = TPS == 1 ? 0 : (int)threadIdx.x / SPI;
  const uint32_t Lt = (uint32_t)S.Lt, L = (uint32_t)S.L;
  VCount<uint32_t, kLanesKs> cs[NH];
  VCount<uint32_t, kLanesKt> ct[NH];
  if (BLUE)
#pragma unroll
    for (int h = 0; h < NH; ++h) {
      cs[h].zero();
      ct[h].zero();
    }

  int n_it = 0;   // sites per thread in the counters
  for (int base = 0; base < n; base += SPI) {
    const bool live = base + sl < n;
    uint32_t site = 0;
    uint32_t sc[NH], P0[NH], P1[NH], P2[NH], Q0[NH], Q1[NH], fw[NH];
#pragma unroll
    for (int h = 0; h < NH; ++h) sc[h] = P0[h] = P1[h] = P2[h] = Q0[h] = Q1[h] = fw[h] = 0;
    if (live) {
      const uint32_t j = (uint32_t)(j0 + base + sl);
      const uint32_t tau = S.hpd.div(j), rem = j - tau * (uint32_t)hp;
      const uint32_t y = S.hld.div(rem), x = 2 * (rem - y * (L >> 1)) + ((y + tau + (uint32_t)colour) & 1u);
      const uint32_t i2 = x + L * y, offt = tau * (uint32_t)plane;
      const uint32_t ixp = x + 1 == L ? i2 + 1 - L : i2 + 1, ixm = x == 0 ? i2 + L - 1 : i2 - 1;
      const uint32_t iyp = y + 1 == L ? x : i2 + L, iym = y == 0 ? i2 + plane - L : i2 - L;
      site = i2 + offt;
      const uint32_t i_tp = i2 + (tau + 1 == Lt ? 0u : offt + plane);
      const uint32_t i_tm = i2 + (tau == 0 ? (Lt - 1) * plane : offt - plane);
      // the antiperiodic wrap bond is unsatisfied when its spins agree
      const uint32_t gtp = ones_if<uint32_t>(S.tau_ap && tau + 1 == Lt), gtm = ones_if<uint32_t>(S.tau_ap && tau == 0);
      const uint32_t jh = S.J[i2];
      const uint32_t Jxp = 0u - (jh & 1u), Jyp = 0u - (jh >> 1), Jxm = 0u - (S.J[ixm] & 1u);
      const uint32_t Jym = 0u - ((uint32_t)S.J[iym] >> 1);
      auto bonds = [&](int h, uint32_t c, uint32_t xp, uint32_t xm, uint32_t yp, uint32_t ym, uint32_t up, uint32_t dn) {
        const uint32_t b1 = c ^ xp ^ Jxp, b2 = c ^ xm ^ Jxm, b3 = c ^ yp ^ Jyp, b4 = c ^ ym ^ Jym;
        const uint32_t t1 = c ^ up ^ gtp, t2 = c ^ dn ^ gtm;
        const uint32_t s1 = b1 ^ b2 ^ b3, c1 = maj3(b1, b2, b3), c2 = s1 & b4;
        sc[h] = c;
        P0[h] = s1 ^ b4;
        P1[h] = c1 ^ c2;
        P2[h] = c1 & c2;
        Q0[h] = t1 ^ t2;
        Q1[h] = t1 & t2;
      };
      if constexpr (TPS == 1) {
#pragma unroll
        for (int g = 0; g < MG; ++g)
          if (g < NG) {
            const Word *w = S.spins + (size_t)g * S.N;
            const Word c = ld_word<CG>(w + site), xp = ld_word<CG>(w + ixp + offt), xm = ld_word<CG>(w + ixm + offt);
            const Word yp = ld_word<CG>(w + iyp + offt), ym = ld_word<CG>(w + iym + offt);
            const Word up = ld_word<CG>(w + i_tp), dn = ld_word<CG>(w + i_tm);
#pragma unroll
            for (int k = 0; k < HW; ++k)
              bonds(g * HW + k, (uint32_t)(c >> (32 * k)), (uint32_t)(xp >> (32 * k)), (uint32_t)(xm >> (32 * k)),
                    (uint32_t)(yp >> (32 * k)), (uint32_t)(ym >> (32 * k)), (uint32_t)(up >> (32 * k)),
                    (uint32_t)(dn >> (32 * k)));
          }
      } else if (part < NG * HW) {   // one half per part (MH <= TPS)
        const int g = part / HW, k = part - g * HW;
        const uint32_t *w = reinterpret_cast<const uint32_t *>(S.spins + (size_t)g * S.N) + k;
        auto ld = [&](uint32_t i) { return ld_word<CG>(w + (size_t)i * HW); };
        bonds(0, ld(site), ld(ixp + offt), ld(ixm + offt), ld(iyp + offt), ld(iym + offt), ld(i_tp), ld(i_tm));
      }
    }
    if (!count_only) {
      if (live) {
#pragma unroll
        for (int h = 0; h < NH; ++h) {
          const int hh = TPS == 1 ? h : part;
          if (hh < NG * HW)
            lanes_store_codes(code_s + ((hh / HW) * 16 + (hh % HW) * 8) * kLanesThreads + sl, P0[h], P1[h], P2[h],
                              Q0[h], Q1[h]);
        }
      }
      if (TPS > 1) __syncthreads();   // the codes of a site come from, and go to, several warps
      Word flips[MG];
#pragma unroll
      for (int g = 0; g < MG; ++g) flips[g] = 0;
      if (live) {
        // Philox rounds 1 and 2 of the site: A, y2 and B depend on it alone
        const uint2 key = S.key;
        const uint32_t z1 = __umulhi(kPhiloxM0, site) ^ S.ctr_w ^ key.y;
        const uint32_t A = __umulhi(kPhiloxM1, z1) ^ (key.x + kPhiloxW0), y2 = kPhiloxM1 * z1;
        const uint32_t B = (kPhiloxM0 * site) ^ (key.y + kPhiloxW1);
        const unsigned char *cb = reinterpret_cast<const unsigned char *>(code_s + sl);
        for (int q = 0; q < nq; ++q) {
          uint32_t f[4] = {0, 0, 0, 0};   // flip bits of the quad's replicas, by walker
#pragma unroll 2
          for (int s = part; s < n_slots; s += TPS) {
            const int e = s * nq + q;
            const uint4 ph = phx[e], i0 = inf[2 * e], i1 = inf[2 * e + 1];
            uint4 c = make_uint4(A ^ ph.x, y2, ph.y ^ B, ph.z);
            uint2 k = make_uint2(key.x + 2 * kPhiloxW0, key.y + 2 * kPhiloxW1);
#pragma unroll
            for (int i = 2; i < 10; ++i) {
              const uint32_t lo0 = kPhiloxM0 * c.x, hi0 = __umulhi(kPhiloxM0, c.x);
              const uint32_t lo1 = kPhiloxM1 * c.z, hi1 = __umulhi(kPhiloxM1, c.z);
              c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
              k.x += kPhiloxW0;
              k.y += kPhiloxW1;
            }
            const unsigned char *row = reinterpret_cast<const unsigned char *>(T16 + s * 16);
            // a draw flips iff R < T or T = 2^32 - 1: with R cut to 2^32 - 2
            // (no finite T exceeds that) both are R < T
            // (with a thread per site the bit is added by a predicated
            // multiply-add, off the logic pipe: the uneven batch 114.8 -> 111.8
            // ms; TPS = 4, which latency bounds, is as fast with an or)
            auto lane = [&](int jj, uint32_t off, uint32_t bit, uint32_t R) {
              const uint32_t thr = *reinterpret_cast<const uint32_t *>(row + cb[off]);
              if constexpr (TPS == 1) add_if_less(f[jj], min(R, 0xFFFFFFFEu), thr, bit, S.one);
              else if (min(R, 0xFFFFFFFEu) < thr) f[jj] |= bit;
            };
            lane(0, i0.x, i0.y, c.x);
            lane(1, i0.z, i0.w, c.y);
            lane(2, i1.x, i1.y, c.z);
            lane(3, i1.z, i1.w, c.w);
          }
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) {
            const int r = 4 * q + jj;
            if (r < n_rep) {
              const int g = MG > 1 && r >= S.rpw ? 1 : 0;   // n_groups <= 2
              const Word m = (Word)f[jj] << ((r - g * S.rpw) * n_slots);
              if (MG > 1 && g) flips[MG - 1] |= m;
              else flips[0] |= m;
            }
          }
        }
      }
      if constexpr (TPS == 1) {
#pragma unroll
        for (int g = 0; g < MG; ++g)
          if (g < NG) {
#pragma unroll
            for (int k = 0; k < HW; ++k) fw[g * HW + k] = (uint32_t)(flips[g] >> (32 * k));
            if (flips[g]) {
              Word c = 0;
#pragma unroll
              for (int k = 0; k < HW; ++k) c |= (Word)(sc[g * HW + k] ^ fw[g * HW + k]) << (32 * k);
              S.spins[(size_t)g * S.N + site] = c;
            }
          }
      } else {
#pragma unroll
        for (int hh = 0; hh < MH; ++hh) fx[hh * kLanesThreads + threadIdx.x] = (uint32_t)(flips[hh / HW] >> (32 * (hh % HW)));
        __syncthreads();
        if (live && part < NG * HW) {
#pragma unroll
          for (int u = 0; u < TPS; ++u) fw[0] |= fx[part * kLanesThreads + u * SPI + sl];
          if (fw[0]) {
            const int g = part / HW, k = part - g * HW;
            reinterpret_cast<uint32_t *>(S.spins + (size_t)g * S.N)[(size_t)site * HW + k] = sc[0] ^ fw[0];
          }
        }
      }
    }
    if (BLUE) {
      // unsatisfied counts after the flip: u -> 4 - u (spatial), 2 - u (tau);
      // threads without a site add zeros
#pragma unroll
      for (int h = 0; h < NH; ++h) {
        const uint32_t f = fw[h];
        cs[h].add3(P0[h], P1[h] ^ (f & P0[h]), mux(f, ~(P0[h] | P1[h] | P2[h]), P2[h]));
        ct[h].add2(Q0[h], mux(f, ~(Q0[h] | Q1[h]), Q1[h]));
      }
      if (++n_it == kLanesFlushSites || base + SPI >= n) {
        // the planes in use (u_s <= 4, u_t <= 2 a site)
        const int ks = 32 - __clz(4 * n_it), kt = ks - 1, lane = threadIdx.x & 31;
#pragma unroll
        for (int h = 0; h < NH; ++h) {
          const int hh = TPS == 1 ? h : part;
          if (hh < NG * HW) {   // uniform over the warp
            int us = 0, ut = 0;
#pragma unroll
            for (int i = 0; i < kLanesKs; ++i)
              if (i < ks) us += __popc(warp_transpose32(cs[h].p[i], lane)) << i;
#pragma unroll
            for (int i = 0; i < kLanesKt; ++i)
              if (i < kt) ut += __popc(warp_transpose32(ct[h].p[i], lane)) << i;
            const int at = (hh / HW) * W + (hh % HW) * 32 + lane;
            if (us) atomicAdd(&acc_s[at], us);
            if (ut) atomicAdd(&acc_t[at], ut);
          }
          cs[h].zero();
          ct[h].zero();
        }
        n_it = 0;
      }
    }
  }
  if (BLUE) {
    __syncthreads();
    for (int i = threadIdx.x; i < NG * W; i += kLanesThreads) {
      const int g = i / W, l = i - g * W;
      const int rl = l / n_slots, w = l - rl * n_slots;
      const int r = g * S.rpw + rl;
      if (rl >= S.rpw || r >= n_rep) continue;
      unsigned long long *u = S.U + ((size_t)r * n_slots + w) * 2;
      if (acc_s[i]) atomicAdd(u, (unsigned long long)acc_s[i]);
      if (acc_t[i]) atomicAdd(u + 1, (unsigned long long)acc_t[i]);
    }
  }
}

}  // namespace qisg
