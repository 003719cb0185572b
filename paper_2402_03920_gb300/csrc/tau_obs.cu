// Imaginary-time observables of the configurations now at each ladder slot
// (Appendix E.1, the quantities of the overlap_tau and corr_euclidea
// programs, computed online on the resident configurations instead of from
// files).  For one configuration S and a lag tau (tau_1 + tau taken modulo
// L_tau):
//   q~_x(tau_1, tau) = S_{x, tau_1} S_{x, tau_1 + tau},
//   Q~(tau_1, tau)   = sum_x q~_x(tau_1, tau),
// and over tau_1 = 0 .. L_tau-1 the sums
//   S1(tau) = sum Q~                  (L^2 L_tau times the site average of C_x(tau))
//   S2(tau) = sum Q~^2, S4(tau) = sum Q~^4    (L_tau Q_2(tau), L_tau Q_4(tau))
//   SF(tau) = sum ( |sum_x e^{i 2 pi x_1 / L} q~_x|^2 + |sum_x e^{i 2 pi x_2 / L} q~_x|^2 )
//                                     (2 L_tau F(tau))
// per (sample, replica, slot); averages over measurements and replicas are
// the caller's.
//
// With C_x the column (or row) sums of q~ and E_x = C_x - C_{x+L/2}, x < L/2,
// the half-period fold of the wave e^{i 2 pi x / L},
//   |sum_x e^{i 2 pi x / L} C_x|^2 = N_0 + 2 sum_{1 <= d < L/4} cos(2 pi d / L) N_d,
//   N_d = sum_{x < L/2} E_x E_{x+d},  E_{x+L/2} = -E_x
// (cos(pi - z) = -cos z joins d and L/2 - d; d = L/4 has cosine 0).  The N_d
// are whole numbers, so they are summed over tau_1, rows and columns exactly
// in integers and the cosines enter once per lag: SF has a few roundings
// where the double sums over x and tau_1 had thousands, and the FP64 unit (2
// lanes an SM) drops out.  All four sums are the same at lags tau and
// L_tau - tau (the same pairs of slices), so lags 1 .. L_tau / 2 are done.
// Where the terms cancel (SF below 1/16 of the sum of their magnitudes, a
// near-uniform q~; always at lag 0, whose SF the host computes) that lag is
// evaluated as written above instead: rows and columns in order x = 0 .. L-1,
// FP64 without contraction, a warp per lag with the tau_1 over its lanes.
//
// What bounds it: the population counts (16 lanes an SM) and integer issue,
// about 140 instructions per pair of slices at L = 16.  A block takes one
// configuration: its spins (staged as int8 by walker) become two bitmaps per
// tau-plane in shared memory, one word per row (fixed x_2, bit x_1) and one
// per column (fixed x_1, bit x_2).  Up to L = 16 a word holds row x and row
// x + L/2 side by side: with the upper half complemented one count gives
// E_x, and the total for Q~ comes from carry-save sums of the words.  A plane's
// words are contiguous with a pitch of an odd number of 16-byte units, so
// that threads at consecutive lags read them as 16-byte words without bank
// conflicts.  A thread owns a lag and a part of the tau_1.  The call on 2048
// configurations at L = 16, L_tau = 256 takes 1.33 ms, 0.46 of it this kernel
// (45.8 ms with the FP64 sums over every lag; 23 to 30 where every lag cancels,
// as in configurations that are constant along tau, FP64 issue again).
#include <algorithm>
#include <cmath>
#include <utility>
#include <vector>

#include "qisg_internal.cuh"

namespace qisg {
namespace {

constexpr int kTauBlock = 256;
constexpr size_t kTauSmemMax = 227 * 1024;

struct TauArgs {
  const int8_t *S;
  const int32_t *walker;
  int64_t a0;
  int n_rep, n_slots, Lt;
  int pitch;                  // words per plane in shared memory
  int parts;                  // threads per lag (each a part of tau_1); 1 when L_tau / 2 > 128
  const double *cs, *sn;
  double sf0;                 // SF at lag 0
  long long *S1, *S2, *S4;
  double *SF;
};

// Population count of N words through full adders (three words to a sum and
// a carry word).
template <int N>
__device__ __forceinline__ int popc_sum(const uint32_t (&w)[N]) {
  if constexpr (N == 0) {
    return 0;
  } else if constexpr (N <= 2) {
    int c = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) c += __popc(w[i]);
    return c;
  } else {
    constexpr int F = N / 3, R = N % 3;
    uint32_t s[F + R], c[F];
#pragma unroll
    for (int i = 0; i < F; ++i) {
      s[i] = w[3 * i] ^ w[3 * i + 1] ^ w[3 * i + 2];
      c[i] = maj3(w[3 * i], w[3 * i + 1], w[3 * i + 2]);
    }
#pragma unroll
    for (int i = 0; i < R; ++i) s[F + i] = w[3 * F + i];
    return popc_sum<F + R>(s) + 2 * popc_sum<F>(c);
  }
}

// The bitmaps of a plane: NW words of columns, then NW words of rows.
template <int L>
struct TauPlane {
  static constexpr int H = L / 2;
  static constexpr bool kPacked = L <= 16;            // word x: row x | row x + L/2 << 16
  static constexpr int NW = kPacked ? H : L;
  static constexpr int kQuads = (2 * NW + 3) / 4;     // 16-byte words read per plane
  __device__ static __forceinline__ uint32_t line(const uint32_t *w, int x) {   // row or column x
    if constexpr (kPacked) return x < H ? w[x] & 0xFFFFu : w[x - H] >> 16;
    else return w[x];
  }
};

// SF of one lag from its definition, by one warp: lane l takes the tau_1
// congruent to l.  Every lane gets the sum.  (Inlined: with a call in it the
// kernel schedules its main loop worse, 499 against 459 us at L = 16, L_tau = 256.)
template <int L>
__device__ __forceinline__ double tau_sf_direct(const TauArgs &a, const uint32_t *W, int tau) {
  using P = TauPlane<L>;
  double sf = 0.0;
  for (int t1 = threadIdx.x & 31; t1 < a.Lt; t1 += 32) {
    const int t2 = t1 + tau < a.Lt ? t1 + tau : t1 + tau - a.Lt;
    const uint32_t *w1 = W + (size_t)t1 * a.pitch, *w2 = W + (size_t)t2 * a.pitch;
    double re1 = 0.0, im1 = 0.0, re2 = 0.0, im2 = 0.0;
    for (int x = 0; x < L; ++x) {
      const int C = L - 2 * __popc(P::line(w1, x) ^ P::line(w2, x));                   // sum over x2 at x1 = x
      const int R = L - 2 * __popc(P::line(w1 + P::NW, x) ^ P::line(w2 + P::NW, x));   // sum over x1 at x2 = x
      re1 = __dadd_rn(re1, __dmul_rn(a.cs[x], (double)C));
      im1 = __dadd_rn(im1, __dmul_rn(a.sn[x], (double)C));
      re2 = __dadd_rn(re2, __dmul_rn(a.cs[x], (double)R));
      im2 = __dadd_rn(im2, __dmul_rn(a.sn[x], (double)R));
    }
    const double f1 = __dadd_rn(__dmul_rn(re1, re1), __dmul_rn(im1, im1));
    const double f2 = __dadd_rn(__dmul_rn(re2, re2), __dmul_rn(im2, im2));
    sf = __dadd_rn(sf, __dadd_rn(f1, f2));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sf = __dadd_rn(sf, __shfl_xor_sync(0xffffffffu, sf, o));
  return sf;
}

template <int L>
__global__ void __launch_bounds__(kTauBlock) tau_obs_kernel(const TauArgs a) {
  using P = TauPlane<L>;
  constexpr int H = P::H, NW = P::NW, D = (H + 1) / 2;
  extern __shared__ __align__(16) uint32_t W[];       // [Lt][pitch]
  const int64_t c = blockIdx.x;                       // configuration (ai, r, s) of this chunk
  const int s = (int)(c % a.n_slots);
  const int64_t ar = c / a.n_slots;                   // ai * n_rep + r
  const int64_t ai = ar / a.n_rep;
  const int r = (int)(ar - ai * a.n_rep);
  const int w = a.walker[((a.a0 + ai) * a.n_rep + r) * a.n_slots + s];
  const int Lt = a.Lt;
  const int8_t *src = a.S + (ar * a.n_slots + w) * ((int64_t)L * L * Lt);
  // rows, two spins per load (a row starts at an even byte)
  for (int i = threadIdx.x; i < Lt * NW; i += kTauBlock) {
    const int tau = i / NW, k = i - tau * NW;
    auto row = [&](int x2) {
      const uint16_t *q = reinterpret_cast<const uint16_t *>(src + (int64_t)L * (x2 + (int64_t)L * tau));
      uint32_t v = 0;
#pragma unroll
      for (int j = 0; j < H; ++j) {
        const uint32_t u = q[j];   // bytes 1 or 0xFF: bit 7 of a byte is the spin bit
        v |= (((u >> 7) & 1u) | ((u >> 14) & 2u)) << (2 * j);
      }
      return v;
    };
    W[(size_t)tau * a.pitch + NW + k] = P::kPacked ? row(k) | (row(k + H) << 16) : row(k);
  }
  __syncthreads();
  // columns: the planes' bitmaps transposed
  for (int i = threadIdx.x; i < Lt * NW; i += kTauBlock) {
    const int tau = i / NW, k = i - tau * NW;
    const uint32_t *rw = W + (size_t)tau * a.pitch + NW;
    uint32_t v = 0;
#pragma unroll
    for (int x2 = 0; x2 < L; ++x2) {
      const uint32_t l = P::line(rw, x2);
      v |= ((l >> k) & 1u) << x2;
      if constexpr (P::kPacked) v |= ((l >> (k + H)) & 1u) << (16 + x2);
    }
    W[(size_t)tau * a.pitch + k] = v;
  }
  __syncthreads();
  const int nl = Lt / 2, per = a.parts;
  constexpr uint32_t kMask = P::kPacked ? ((1u << L) - 1u) << 16 : 0u;
  int *red = reinterpret_cast<int *>(W + (size_t)Lt * a.pitch);   // parts > 1: [D + 2][kTauBlock], then S4
  bool left = false;   // a lag of this thread cancels
  for (int lag0 = 0; lag0 < nl; lag0 += kTauBlock / per) {
    const int lanes = min(nl - lag0, kTauBlock / per);
    const int part = (int)threadIdx.x / lanes;
    const int tau = 1 + lag0 + (int)threadIdx.x - part * lanes;
    const bool live = part < per;
    int nd[D], s1 = 0;
    uint32_t s2 = 0;
    unsigned long long s4 = 0;
#pragma unroll
    for (int d = 0; d < D; ++d) nd[d] = 0;
    if (live) {
      const int lo = part * Lt / per, hi = (part + 1) * Lt / per;
      for (int t1 = lo; t1 < hi; ++t1) {
        const int t2 = t1 + tau < Lt ? t1 + tau : t1 + tau - Lt;
        const uint4 *w1 = reinterpret_cast<const uint4 *>(W + (size_t)t1 * a.pitch);
        const uint4 *w2 = reinterpret_cast<const uint4 *>(W + (size_t)t2 * a.pitch);
        uint32_t y[4 * P::kQuads];
#pragma unroll
        for (int i = 0; i < P::kQuads; ++i) {
          const uint4 u = w1[i], v = w2[i];
          y[4 * i] = u.x ^ v.x;
          y[4 * i + 1] = u.y ^ v.y;
          y[4 * i + 2] = u.z ^ v.z;
          y[4 * i + 3] = u.w ^ v.w;
        }
        int down = 0;   // sites where q~ = -1
        if constexpr (P::kPacked) {
          uint32_t rows[NW];
#pragma unroll
          for (int x = 0; x < NW; ++x) rows[x] = y[NW + x];
          down = popc_sum<NW>(rows);
        }
#pragma unroll
        for (int axis = 0; axis < 2; ++axis) {
          int e[H];   // -E_x / 2
#pragma unroll
          for (int x = 0; x < H; ++x) {
            const uint32_t *z = y + axis * NW;
            if constexpr (P::kPacked) {
              e[x] = __popc(z[x] ^ kMask) - L;
            } else {
              const int p0 = __popc(z[x]), p1 = __popc(z[x + H]);
              e[x] = p0 - p1;
              if (axis == 1) down += p0 + p1;
            }
          }
#pragma unroll
          for (int d = 0; d < D; ++d)
#pragma unroll
            for (int x = 0; x < H; ++x) nd[d] += x + d < H ? e[x] * e[x + d] : e[x] * -e[x + d - H];
        }
        const int q = L * L - 2 * down;
        const uint32_t q2 = (uint32_t)(q * q);
        s1 += q;
        s2 += q2;   // L^4 L_tau < 2^31: 8 L L_tau bytes fit shared memory
        s4 += (unsigned long long)q2 * q2;
      }
    }
    if (per > 1) {
      unsigned long long *red4 = reinterpret_cast<unsigned long long *>(red + (D + 2) * kTauBlock);
      __syncthreads();
      if (live) {
#pragma unroll
        for (int d = 0; d < D; ++d) red[d * kTauBlock + threadIdx.x] = nd[d];
        red[D * kTauBlock + threadIdx.x] = s1;
        red[(D + 1) * kTauBlock + threadIdx.x] = (int)s2;
        red4[threadIdx.x] = s4;
      }
      __syncthreads();
      if (part == 0)
        for (int u = 1; u < per; ++u) {
          const int o = u * lanes + threadIdx.x;
#pragma unroll
          for (int d = 0; d < D; ++d) nd[d] += red[d * kTauBlock + o];
          s1 += red[D * kTauBlock + o];
          s2 += (uint32_t)red[(D + 1) * kTauBlock + o];
          s4 += red4[o];
        }
    }
    if (part == 0) {
      double sf = (double)nd[0], mag = (double)nd[0];
#pragma unroll
      for (int d = 1; d < D; ++d) {
        const double v = __dmul_rn(2.0 * a.cs[d], (double)nd[d]);
        sf = __dadd_rn(sf, v);
        mag = __dadd_rn(mag, fabs(v));
      }
      const bool direct = !(16.0 * sf > mag);
      left |= direct;
      for (int k = 0; k < 2; ++k) {   // lags tau and L_tau - tau
        const int lag = k ? Lt - tau : tau;
        if (k && lag == tau) break;
        const int64_t o = c * Lt + lag;
        a.S1[o] = s1;
        a.S2[o] = (long long)s2;
        a.S4[o] = (long long)s4;
        a.SF[o] = direct ? -1.0 : 4.0 * sf;   // -1 (no SF is negative): left to a warp below
      }
    }
  }
  // the lags whose terms cancel, a warp each; tau and L_tau - tau have the same terms
  if (__syncthreads_or(left))
    for (int tau = 1 + (int)(threadIdx.x >> 5); tau <= nl; tau += kTauBlock / 32) {
      double *o = a.SF + c * Lt;
      if (o[tau] >= 0.0) continue;   // the same in every lane
      const double sf = tau_sf_direct<L>(a, W, tau);
      __syncwarp();                  // every lane has read the mark
      if ((threadIdx.x & 31) == 0) o[tau] = o[Lt - tau] = sf;
    }
  if (threadIdx.x == 0) {   // lag 0: q~ = 1 at every site
    const int64_t o = c * Lt;
    const long long q = (long long)L * L;
    a.S1[o] = q * Lt;
    a.S2[o] = q * q * Lt;
    a.S4[o] = q * q * q * q * Lt;
    a.SF[o] = a.sf0;
  }
}

// Launch for lattice side L (even, 2 .. 32).
template <int L>
int launch_tau(int l, const TauArgs &a, unsigned blocks, cudaStream_t st) {
  if (l != L) {
    if constexpr (L < 32) return launch_tau<L + 2>(l, a, blocks, st);
    else return fail(QISG_EINVAL, "tau observables take L <= 32");
  } else {
    using P = TauPlane<L>;
    TauArgs b = a;
    // an odd number of 16-byte units per plane while that fits
    const int tight = P::kQuads, odd = tight | 1;
    const size_t cap = kTauSmemMax;
    b.pitch = 4 * ((size_t)odd * 16 * a.Lt <= cap ? odd : tight);
    b.parts = std::max(1, kTauBlock / std::max(1, a.Lt / 2));
    size_t smem = (size_t)b.pitch * 4 * a.Lt;
    constexpr size_t kRed = ((P::H + 1) / 2 + 2) * kTauBlock * 4 + kTauBlock * 8;
    if (b.parts > 1) smem += kRed;   // L_tau <= 256: fits
    if (smem > 48 * 1024) {   // one limit for all callers: threads with other L_tau may be between this and their launch
      const int rc = cuda_check(cudaFuncSetAttribute(tau_obs_kernel<L>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                     (int)kTauSmemMax),
                                "shared memory");
      if (rc) return rc;
    }
    tau_obs_kernel<L><<<blocks, kTauBlock, smem, st>>>(b);
    return cuda_check(cudaGetLastError(), "tau observables");
  }
}

}  // namespace
}  // namespace qisg

using namespace qisg;

extern "C" int qisg_tau_observables(qisg_handle *h, int64_t a_lo, int64_t n_a, int64_t *S1, int64_t *S2,
                                    int64_t *S4, double *SF) {
  if (!h || ((!S1 || !S2 || !S4 || !SF) && n_a > 0)) return fail(QISG_EINVAL, "NULL argument");
  if (a_lo < 0 || n_a < 0 || a_lo + n_a > h->n_samples) return fail(QISG_EINVAL, "sample range");
  if (h->L > 32) return fail(QISG_EINVAL, "tau observables take L <= 32");
  const size_t smem = (size_t)2 * h->Lt * h->L * 4;
  if (smem > kTauSmemMax) return fail(QISG_EINVAL, "tau observables: 2 L L_tau words exceed shared memory");
  if (n_a == 0) return QISG_OK;
  int rc = handle_sync(h);
  if (rc) return rc;
  // cos / sin of 2 pi x / L, x = 0 .. L-1 (host libm, FP64)
  std::vector<double> tab((size_t)2 * h->L);
  for (int x = 0; x < h->L; ++x) {
    tab[(size_t)x] = std::cos(2.0 * M_PI * x / h->L);
    tab[(size_t)h->L + x] = std::sin(2.0 * M_PI * x / h->L);
  }
  const int64_t per_a = (int64_t)h->n_rep * h->n_slots * h->N;
  const int64_t cfg_a = (int64_t)h->n_rep * h->n_slots;
  const int64_t chunk = std::min(n_a, std::max<int64_t>(1, ((int64_t)256 << 20) / per_a));
  int8_t *stage = nullptr;
  double *d_tab = nullptr;
  long long *d_out = nullptr;   // S1, S2, S4 of a chunk, then SF
  const size_t n_out = (size_t)(chunk * cfg_a * h->Lt);
  rc = cuda_check(cudaMalloc(&stage, (size_t)(chunk * per_a)), "cudaMalloc");
  if (!rc) rc = cuda_check(cudaMalloc(&d_tab, tab.size() * 8), "cudaMalloc");
  if (!rc) rc = cuda_check(cudaMalloc(&d_out, n_out * 4 * 8), "cudaMalloc");
  if (!rc) rc = cuda_check(cudaMemcpyAsync(d_tab, tab.data(), tab.size() * 8, cudaMemcpyHostToDevice, h->stream),
                           "copy table");
  // lag 0: every column and row sum is L
  double sf0 = 0.0;
  {
    double re = 0.0, im = 0.0;
    for (int x = 0; x < h->L; ++x) {
      re = re + tab[(size_t)x] * (double)h->L;
      im = im + tab[(size_t)h->L + x] * (double)h->L;
    }
    const double f = re * re + im * im;
    for (int t1 = 0; t1 < h->Lt; ++t1) sf0 = sf0 + (f + f);
  }
  for (int64_t a0 = 0; a0 < n_a && !rc; a0 += chunk) {
    const int64_t na = std::min(chunk, n_a - a0), nc = na * cfg_a, no = nc * h->Lt;
    rc = h->layout == QISG_LAYOUT_LANES   ? lanes_stage_spins(h, a_lo + a0, na, stage)
         : h->layout == QISG_LAYOUT_SITES ? sites_stage_spins(h, a_lo + a0, na, stage)
                                          : samples_stage_spins(h, a_lo + a0, na, stage);
    if (rc) break;
    TauArgs args{stage, h->d_walker, a_lo + a0, h->n_rep, h->n_slots, h->Lt, 0, 1, d_tab, d_tab + h->L, sf0,
                 d_out, d_out + n_out, d_out + 2 * n_out, reinterpret_cast<double *>(d_out + 3 * n_out)};
    rc = launch_tau<2>(h->L, args, (unsigned)nc, h->stream);
    h->launches++;
    const int64_t o = a0 * cfg_a * h->Lt;
    if (!rc) rc = cuda_check(cudaMemcpyAsync(S1 + o, d_out, (size_t)no * 8, cudaMemcpyDeviceToHost, h->stream), "copy");
    if (!rc)
      rc = cuda_check(cudaMemcpyAsync(S2 + o, d_out + n_out, (size_t)no * 8, cudaMemcpyDeviceToHost, h->stream), "copy");
    if (!rc)
      rc = cuda_check(cudaMemcpyAsync(S4 + o, d_out + 2 * n_out, (size_t)no * 8, cudaMemcpyDeviceToHost, h->stream),
                      "copy");
    if (!rc)
      rc = cuda_check(cudaMemcpyAsync(SF + o, d_out + 3 * n_out, (size_t)no * 8, cudaMemcpyDeviceToHost, h->stream),
                      "copy");
    if (!rc) rc = handle_sync(h);
  }
  if (stage) cudaFree(stage);
  if (d_tab) cudaFree(d_tab);
  if (d_out) cudaFree(d_out);
  return rc;
}
