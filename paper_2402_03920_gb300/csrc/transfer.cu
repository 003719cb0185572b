// The transfer-matrix product of the exact-diagonalisation code (Sec. 2.2,
// Eq. (transfer-matrix); Appendix D), on one GPU for L <= 5: out = T in on
// the even or odd parity sector, vectors of 2^{L^2-1} doubles indexed by the
// parity-aware basis |n>_{e,o}.
//
//   psi[n] = in[n] w[n];   rounds j = 0 .. L^2-2: psi[n] <- jP psi[n] + jM psi[n ^ 2^j];
//   last factor (Eq. (lr)): psi[n] <- jP psi[n] + parity jM psi[2^{L^2-1} - 1 - n];
//   out[n] = psi[n] w[n],
// with w[n] = exp((k/2) sum_bonds J S S) of n read as an L^2-bit spin
// configuration (top bit 0), jP = e^{k_tau} / (e^{k_tau} + e^{-k_tau}) and
// jM = e^{-k_tau} / (...)  (Eq. (expH1) with exp(-2 k_tau) = tanh(k Gamma)).
//
// What bounds it: FP64 issue (about 0.62e12 FP64 operations a second here;
// the vector crosses HBM three times at L = 5, 0.12 ms of 6.8 TB/s).  So the
// rounds are taken with the factor jP outside: with r = jM / jP a pair update
// is x' = x + r y, y' = y + r x, one fused multiply-add per element, and jP^{L^2}
// goes into the table of w used on load.  (jP x + jM y as y + jP (x - y) takes
// three operations per pair: 1.351 ms at L = 5 in that form, 0.889 now.)  This is the
// paper's formula rearranged: the results differ by rounding only (relative
// 1e-15 in norm after 25 rounds), and the scaled values stay below the
// plain ones until the last round.
//
// Rounds are fused in tiles so that the vector crosses HBM once per pass
// instead of once per round: a tile fixes all index bits except a low run
// [0, c) (c = 5: 32 consecutive doubles, 256-byte segments) and the bits
// [lo, hi) of the pass's rounds; the first pass takes bits [0, 12) whole.
// Within a tile a thread takes up to three rounds on 8 elements in registers
// (in the last pass on 8 and their complement's 8), so shared memory is
// crossed once per three rounds and, where the run of low bits makes
// a warp's accesses whole segments, the first group reads HBM and the last
// group writes it directly.  The last pass pairs every tile with its bit
// complement (the tile holding 2^{n} - 1 - n for each n) for the parity
// factor, again in registers.  w is not stored: each thread computes the bond
// energy of its index with bit rotations and popcounts and looks exp((k/2) E)
// up in a table of the 2 L^2 + 1 possible energies, computed once on the host
// in FP64.  Rounds run in ascending j for every element, as in the paper.
#include <cmath>
#include <vector>

#include "qisg_internal.cuh"

namespace qisg {
namespace {

constexpr int kTransferBlock = 256;
constexpr int kTileLog = 12;   // 4096 doubles, 32 KB of shared memory

struct TransferArgs {
  double r, pr;               // jM / jP and parity times it
  double jPn;                 // jP^{L^2}
  double wtab[51];            // exp((k/2) E) for E = -2 L^2, -2 L^2 + 2, ..., 2 L^2 (L <= 5)
  int L2;                     // L^2
  int sumJ;                   // sum of the couplings
  uint32_t row_last;          // sites with x1 = L-1
  uint32_t not_row_last;      // sites with x1 < L-1 within the lattice
  uint32_t col_last;          // sites with x2 = L-1
  uint32_t not_col_last;      // sites with x2 < L-1
  uint32_t jxp, jxn, jyp, jyn;   // bonds to +x / +y with J = +1 / -1
  int L;
};

// Table index of the L^2-bit configuration n (bit i set <=> S_i = -1):
// E = sum_bonds J S S = sum J - 2 (sum of J over unsatisfied bonds).
__device__ __forceinline__ int energy_index(const TransferArgs &a, uint32_t n) {
  const int L = a.L;
  const uint32_t vx = ((n >> 1) & a.not_row_last) | ((n << (L - 1)) & a.row_last);          // spin at (x1+1, x2)
  const uint32_t vy = ((n >> L) & a.not_col_last) | ((n << (L * (L - 1))) & a.col_last);    // spin at (x1, x2+1)
  const uint32_t ux = n ^ vx, uy = n ^ vy;                                                    // unsatisfied bonds
  const int s = __popc(ux & a.jxp) - __popc(ux & a.jxn) + __popc(uy & a.jyp) - __popc(uy & a.jyn);
  const int E = a.sumJ - 2 * s;
  return (E + 2 * a.L2) >> 1;
}

// One pass: the tile's geometry and what the pass does besides its rounds.
struct PassArgs {
  int c, lo, hi;      // tile bits: [0, c) and the rounds' bits [lo, hi)
  int first;          // multiply by w on load
  int nb;             // index bits
};

// Global index of tile element t: bits [0, c) of t -> bits [0, c), the next
// (hi - lo) bits -> bits [lo, hi), the fixed bits f -> [c, lo) then [hi, nb).
__device__ __forceinline__ uint32_t tile_index(const PassArgs &q, uint32_t t, uint32_t f) {
  const uint32_t low = t & ((1u << q.c) - 1u);
  const uint32_t mid = t >> q.c;
  const uint32_t f_lo = f & ((1u << (q.lo - q.c)) - 1u);   // bits [c, lo)
  const uint32_t f_hi = f >> (q.lo - q.c);                  // bits [hi, nb)
  return low | (f_lo << q.c) | (mid << q.lo) | (f_hi << q.hi);
}

// Shared-memory place of tile element t: one double of padding per 16, so
// that threads reading 8 consecutive elements each meet different banks.
__device__ __forceinline__ uint32_t padded(uint32_t t) { return t + (t >> 4); }

// G rounds on 2^G elements held in registers.
template <int G>
__device__ __forceinline__ void rounds(double (&v)[1 << G], double r) {
#pragma unroll
  for (int b = 0; b < G; ++b)
#pragma unroll
    for (int i = 0; i < (1 << G); ++i)
      if (!(i & (1 << b))) {
        const double x = v[i], y = v[i | (1 << b)];
        v[i] = __fma_rn(r, y, x);
        v[i | (1 << b)] = __fma_rn(r, x, y);
      }
}

// G rounds on tile bits [tb, tb + G) of the whole tile (PAIR: of the tile and
// its complement, element t of the one with element T - 1 - t of the other).
// FROM / TO: elements come from src / go to dst instead of shared memory.
template <int G, bool PAIR, bool FROM, bool TO>
__device__ __forceinline__ void stage(const double *src, double *dst, double *tile, const double *wt,
                                      const TransferArgs &a, const PassArgs &q, int T_log, uint32_t f, int tb) {
  constexpr int M = 1 << G;
  const uint32_t T = 1u << T_log, top = (1u << q.nb) - 1u;
  for (uint32_t p = threadIdx.x; p < T >> G; p += blockDim.x) {
    const uint32_t t0 = ((p >> tb) << (tb + G)) | (p & ((1u << tb) - 1u));
    double v[M], w[PAIR ? M : 1];
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const uint32_t t = t0 | ((uint32_t)m << tb);
      if constexpr (FROM) {
        const uint32_t i = tile_index(q, t, f);
        v[m] = src[i];
        if constexpr (PAIR) w[m] = src[top - i];
      } else {
        v[m] = tile[padded(t)];
        if constexpr (PAIR) w[m] = tile[padded(T + (T - 1u - t))];
      }
    }
    if constexpr (FROM)
      if (q.first) {
#pragma unroll
        for (int m = 0; m < M; ++m) {
          const uint32_t i = tile_index(q, t0 | ((uint32_t)m << tb), f);
          v[m] = __dmul_rn(v[m], wt[energy_index(a, i)]);
          if constexpr (PAIR) w[m] = __dmul_rn(w[m], wt[energy_index(a, top - i)]);
        }
      }
    rounds<G>(v, a.r);
    if constexpr (PAIR) rounds<G>(w, a.r);   // the complement's bit pairs are this one's, swapped
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const uint32_t t = t0 | ((uint32_t)m << tb);
      if constexpr (TO && PAIR) {
        const uint32_t i = tile_index(q, t, f);
        dst[i] = __dmul_rn(__fma_rn(a.pr, w[m], v[m]), wt[64 + energy_index(a, i)]);
        dst[top - i] = __dmul_rn(__fma_rn(a.pr, v[m], w[m]), wt[64 + energy_index(a, top - i)]);
      } else if constexpr (TO) {
        dst[tile_index(q, t, f)] = v[m];
      } else {
        tile[padded(t)] = v[m];
        if constexpr (PAIR) tile[padded(T + (T - 1u - t))] = w[m];
      }
    }
  }
}

template <bool PAIR, bool FROM, bool TO>
__device__ __forceinline__ void stage_g(int g, const double *src, double *dst, double *tile, const double *wt,
                                        const TransferArgs &a, const PassArgs &q, int T_log, uint32_t f, int tb) {
  switch (g) {
    case 1: stage<1, PAIR, FROM, TO>(src, dst, tile, wt, a, q, T_log, f, tb); break;
    case 2: stage<2, PAIR, FROM, TO>(src, dst, tile, wt, a, q, T_log, f, tb); break;
    default: stage<3, PAIR, FROM, TO>(src, dst, tile, wt, a, q, T_log, f, tb); break;
  }
}

// Block f takes the tile of fixed bits f (PAIR, the last pass: and its
// complement, f below half of them).  src and dst may be the same: every
// element is read by the block that writes it, before it does.
template <bool PAIR>
__global__ void __launch_bounds__(kTransferBlock) transfer_pass_kernel(const double *src, double *dst,
                                                                       const __grid_constant__ TransferArgs a,
                                                                       const PassArgs q) {
  extern __shared__ double smem[];
  double *wt = smem, *tile = smem + 128;   // w on load (scaled by jP^{L^2}), w at the end; then the tile(s)
  const int T_log = q.c + (q.hi - q.lo);
  const uint32_t T = 1u << T_log, f = blockIdx.x;
  if (threadIdx.x < 51) {
    wt[threadIdx.x] = __dmul_rn(a.wtab[threadIdx.x], a.jPn);
    wt[64 + threadIdx.x] = a.wtab[threadIdx.x];
  }
  __syncthreads();
  // three rounds on 8 elements a thread, fewer where that would leave less than
  // four warps at work (the last pass at L = 4).  A call at L = 4 | 5: 26.8 | 912 us;
  // four rounds in the unpaired passes 27.7 | 925, three everywhere 27.8 | 911
  const int GM = min(3, max(1, T_log - 7));
  int tb = q.c, left = q.hi - q.lo;
  bool loaded = false;
  if (!PAIR && tb < 4) {   // consecutive elements per thread: load whole segments first
    for (uint32_t t = threadIdx.x; t < T; t += blockDim.x) {
      const uint32_t i = tile_index(q, t, f);
      const double x = src[i];
      tile[padded(t)] = q.first ? __dmul_rn(x, wt[energy_index(a, i)]) : x;
    }
    loaded = true;
    __syncthreads();
  }
  while (left > 0) {
    const int g = left < GM ? left : GM;
    const bool end = left == g;   // the last group writes HBM
    if (!loaded && end)
      stage_g<PAIR, true, true>(g, src, dst, tile, wt, a, q, T_log, f, tb);
    else if (!loaded)
      stage_g<PAIR, true, false>(g, src, dst, tile, wt, a, q, T_log, f, tb);
    else if (end)
      stage_g<PAIR, false, true>(g, src, dst, tile, wt, a, q, T_log, f, tb);
    else
      stage_g<PAIR, false, false>(g, src, dst, tile, wt, a, q, T_log, f, tb);
    loaded = true;
    tb += g;
    left -= g;
    if (!end) __syncthreads();
  }
}

// L = 2 and 3, at most 256 elements: the product in one block, element n in
// thread n, the rounds within a warp by shuffles.  Latency is all there is: the
// kernel takes 2.6 and 3.5 us under ncu (6.2 and 11.2 in the tiled form, whose
// groups of four rounds leave one and 16 threads at work); a call that is waited
// for went from 25 and 28 us to 22 and 23.
__global__ void __launch_bounds__(256) transfer_small_kernel(const double *in, double *out,
                                                             const __grid_constant__ TransferArgs a, int nb) {
  __shared__ double x[256];
  const uint32_t n = threadIdx.x, T = 1u << nb;
  const bool live = n < T;   // L = 2: 8 of a warp
  const double w = live ? a.wtab[energy_index(a, n)] : 0.0;
  double v = live ? __dmul_rn(in[n], __dmul_rn(w, a.jPn)) : 0.0;
  for (int j = 0; j < min(nb, 5); ++j) v = __fma_rn(a.r, __shfl_xor_sync(0xffffffffu, v, 1 << j), v);
  for (int j = 5; j < nb; ++j) {
    x[n] = v;
    __syncthreads();
    v = __fma_rn(a.r, x[n ^ (1u << j)], v);
    __syncthreads();
  }
  x[n] = v;
  __syncthreads();
  if (live) out[n] = __dmul_rn(__fma_rn(a.pr, x[T - 1u - n], v), w);
}

struct Pass {
  int lo, hi, c;
};

// Passes over the rounds: the first takes bits [0, 12) whole; later ones a
// 32-element run of low bits and up to 12 - 5 round bits; the last pass
// holds a tile and its complement, so its tile is at most half as large.
std::vector<Pass> plan_passes(int nb) {
  std::vector<Pass> out;
  int lo = 0;
  while (lo < nb) {
    const int c = lo == 0 ? 0 : (lo < 5 ? lo : 5);
    int w = std::min(nb - lo, kTileLog - c);
    if (lo + w == nb && c + w < nb) w = std::min(w, kTileLog - 1 - c);   // paired tiles
    out.push_back(Pass{lo, lo + w, c});
    lo += w;
  }
  return out;
}

}  // namespace
}  // namespace qisg

using namespace qisg;

extern "C" int qisg_transfer_matvec(const double *in, double *out, int L, double k, double k_tau, const int8_t *J,
                                    int parity, void *cuda_stream) {
  if (!in || !out || !J) return fail(QISG_EINVAL, "NULL argument");
  if (L < 2 || L > 5) return fail(QISG_EINVAL, "transfer matvec takes 2 <= L <= 5 on one GPU");
  if (parity != 1 && parity != -1) return fail(QISG_EINVAL, "parity must be +1 (even) or -1 (odd)");
  if (!std::isfinite(k) || !std::isfinite(k_tau) || k < 0 || k_tau < 0)
    return fail(QISG_EINVAL, "couplings must be finite and >= 0");
  if ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 7u)
    return fail(QISG_EINVAL, "vectors must be 8-byte aligned");
  const int L2 = L * L, nb = L2 - 1;
  TransferArgs a{};
  const double ek = std::exp(k_tau), emk = std::exp(-k_tau);
  const double jP = ek / (ek + emk), jM = emk / (ek + emk);
  a.r = jM / jP;
  a.pr = (double)parity * a.r;
  a.jPn = std::pow(jP, (double)L2);
  for (int e = -2 * L2, i = 0; e <= 2 * L2; e += 2, ++i) a.wtab[i] = std::exp(0.5 * k * (double)e);
  a.L2 = L2;
  a.L = L;
  for (int x2 = 0; x2 < L; ++x2)
    for (int x1 = 0; x1 < L; ++x1) {
      const int i = x1 + L * x2;
      const int jx = J[2 * i], jy = J[2 * i + 1];
      if ((jx != 1 && jx != -1) || (jy != 1 && jy != -1)) return fail(QISG_EINVAL, "couplings must be +-1");
      a.sumJ += jx + jy;
      (x1 == L - 1 ? a.row_last : a.not_row_last) |= 1u << i;
      (x2 == L - 1 ? a.col_last : a.not_col_last) |= 1u << i;
      (jx > 0 ? a.jxp : a.jxn) |= 1u << i;
      (jy > 0 ? a.jyp : a.jyn) |= 1u << i;
    }
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  if (L <= 3) {
    transfer_small_kernel<<<1, std::max(32, 1 << nb), 0, st>>>(in, out, a, nb);
    return cuda_check(cudaGetLastError(), "transfer matvec");
  }
  const std::vector<Pass> plan = plan_passes(nb);
  int rc = QISG_OK;
  for (size_t p = 0; p < plan.size() && !rc; ++p) {
    const Pass &q = plan[p];
    const int width = q.c + (q.hi - q.lo);
    const int fixed = nb - width;
    const bool pair = p + 1 == plan.size();   // the last pass
    const unsigned blocks = pair ? 1u << (fixed - 1) : 1u << fixed;
    const size_t T = (size_t)1 << width, smem = (128 + (pair ? 2 * T + 2 * T / 16 : T + T / 16)) * sizeof(double);
    const PassArgs pa{q.c, q.lo, q.hi, p == 0, nb};
    if (pair)
      transfer_pass_kernel<true><<<blocks, kTransferBlock / 2, smem, st>>>(p == 0 ? in : out, out, a, pa);
    else
      transfer_pass_kernel<false><<<blocks, kTransferBlock, smem, st>>>(p == 0 ? in : out, out, a, pa);
    rc = cuda_check(cudaGetLastError(), "transfer matvec");
  }
  return rc;
}
