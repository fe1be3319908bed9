// Nested slice sampling (Sec. 4.3) on the GPU, around sed_loglike.
//
// Nested sampling (Skilling 2006) keeps n live points drawn from the prior
// inside a rising likelihood contour.  Each iteration here removes the k live
// points of lowest lnL, adds them to the evidence sum, and replaces them by k
// hit-and-run slice chains run side by side: a chain starts at a random
// surviving live point above the contour and makes a fixed number of slice
// steps (Neal 2003: a bracket placed at random around the point, stepped out
// until both ends leave the contour, then shrunk towards the point until a
// proposal lands inside) along directions drawn from the surviving live
// points' covariance.  All chains advance together in rounds: a round kernel
// consumes the last round's likelihoods, moves every chain's state machine on
// to its next proposal and writes the proposals as parameter rows, and one
// sed_loglike call evaluates them.  Proposals that leave the unit cube of the
// box prior are outside the contour without an evaluation.
//
// Prior volume: removing the j-th lowest of n live points shrinks the volume
// by exp(-1 / (n - j)), the expectation of its log shrinkage; the removed
// point's weight is the volume it leaves behind.  Evidence and information take
// an iteration's points at once: FP64 sums over the block in a fixed order, every
// term scaled by the largest (Skilling's recurrence for H after all of them), so
// a run is deterministic for a given seed.
#include <math.h>
#include <string.h>

#include <vector>

#include "sed_internal.cuh"

using namespace sed;

namespace {

constexpr int NSS_MAX_D = 1024;      // parameter columns of a row
constexpr int NSS_FULL_COV = 128;    // full covariance up to this many columns, its diagonal above
constexpr int NSS_MAX_LIVE = 4096;
constexpr int MAXOUT = 16;           // stepping-out moves per side and slice step
constexpr int MAXSHRINK = 48;        // shrinking proposals per slice step (then the step keeps its point)
constexpr int ROUNDS = 16;           // rounds queued between two checks by the host
constexpr int CHAINS_PER_BLOCK = 4;  // one warp per chain

enum Phase : int { PH_NEW = 0, PH_LEFT = 1, PH_RIGHT = 2, PH_SHRINK = 3, PH_DONE = 4 };
enum Tag : uint32_t { TAG_INIT = 1, TAG_START = 2, TAG_DIR = 3, TAG_SLICE = 4 };

struct NssState {
  double lnX, lnZ, H, lstar;
  unsigned long long n_like;
  int n_dead, stop, n_above, pad;
  int active[2];
};

struct Chains {
  float* x0;        // [k][d] current point (unit cube)
  float* v;         // [k][d] direction of the current slice step
  double* lnl0;     // [k] lnL at x0
  float *tL, *tR, *t;
  int *phase, *step, *nl, *nr, *ns, *pend;
  uint32_t* draw;   // per-chain counter of random draws within the iteration
};

struct Live {
  float* U;         // [n][d] unit-cube coordinates
  float* TH;        // [n][d] parameter rows
  double* lnl;      // [n]
  int* order;       // [n] indices in increasing lnL (ties by index)
};

struct Dead {
  float* TH;        // [cap][d]
  double* lnl;      // [cap]
  double* lnw;      // [cap] ln prior weight, turned into the ln posterior weight at the end
  int* rank;        // [cap] insertion ranks
  int cap;
};

// ---- Philox4x32-10 (Salmon, Moraes, Dror & Shaw 2011), counter -> 4 words
__device__ __forceinline__ uint4 philox(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return c;
}
// uniform in (0, 1) from the top 24 bits
__device__ __forceinline__ float u01(uint32_t x) { return ((float)(x >> 8) + 0.5f) * (1.0f / 16777216.0f); }

// Sum (or maximum) of v over the block's first RED_THREADS threads in a fixed
// order, the result in every thread; red holds one value per warp.  (An FP64
// instruction of a warp takes 16 cycles of the SM's pipe on this GPU, so that
// all 32 warps of a block would wait for one another.)
constexpr int RED_THREADS = 256;
template <bool MAX>
__device__ double block_reduce(double v, double* red) {
  auto tree = [](double x, int o0) {
    for (int o = o0; o; o >>= 1) {
      const double w = __shfl_xor_sync(0xffffffffu, x, o);
      x = MAX ? fmax(x, w) : x + w;
    }
    return x;
  };
  if (threadIdx.x < RED_THREADS) {
    v = tree(v, 16);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    v = tree(red[threadIdx.x & (RED_THREADS / 32 - 1)], RED_THREADS / 64);
    __syncwarp();
    if (threadIdx.x == 0) red[0] = v;
  }
  __syncthreads();
  v = red[0];
  __syncthreads();
  return v;
}
// the points of thread j's share of a reduction: j, j + RED_THREADS, ...
__device__ __forceinline__ int red_start(int cnt) { return threadIdx.x < RED_THREADS ? (int)threadIdx.x : cnt; }

// Skilling's update of ln Z and H for the removed points j < cnt of likelihood
// lnl(j) and ln weight lnw(j), by the whole block at once.  Point by point it
// is Z' = Z + w L and H' + ln Z' = (w L ln L + Z (H + ln Z)) / Z'; after all of
// them, with every term scaled by the largest one, Z' = Z + sum w L and
// H' + ln Z' = (Z (H + ln Z) + sum w L ln L) / Z'.  (One thread going through
// the points waited on four FP64 exponentials or logarithms a point.)
template <class Lnl, class Lnw>
__device__ void add_points(NssState* st, int cnt, Lnl lnl, Lnw lnw, double* red) {
  const double lz0 = st->lnZ, h0 = st->H;
  double m = threadIdx.x == 0 ? lz0 : -INFINITY;
  for (int j = red_start(cnt); j < cnt; j += RED_THREADS) m = fmax(m, lnw(j) + lnl(j));
  m = block_reduce<true>(m, red);
  if (m == -INFINITY) return;   // no point with a likelihood yet
  double z = 0.0, u = 0.0;
  if (threadIdx.x == 0 && lz0 > -INFINITY) {
    z = exp(lz0 - m);
    u = z * (h0 + lz0);
  }
  for (int j = red_start(cnt); j < cnt; j += RED_THREADS) {
    const double l = lnl(j);
    if (l == -INFINITY) continue;
    const double e = exp(lnw(j) + l - m);
    z += e;
    u += e * l;
  }
  z = block_reduce<false>(z, red);
  u = block_reduce<false>(u, red);
  if (threadIdx.x == 0) {
    const double lz = m + log(z);
    st->lnZ = lz;
    st->H = u / z - lz;
  }
}

__global__ void k_nss_init(int n, int d, const double* lo, const double* hi, Live lv, NssState* st, uint32_t k0,
                           uint32_t k1) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) {
    st->lnX = 0.0; st->lnZ = -INFINITY; st->H = 0.0; st->lstar = -INFINITY;
    st->n_like = 0; st->n_dead = 0; st->stop = 0; st->n_above = 0;
    st->active[0] = st->active[1] = 0;
  }
  if (i >= n * d) return;
  const int p = i / d, j = i - p * d;
  const uint4 r = philox(make_uint4((uint32_t)p, (uint32_t)(j >> 2), 0u, TAG_INIT), k0, k1);
  const uint32_t w = (j & 3) == 0 ? r.x : (j & 3) == 1 ? r.y : (j & 3) == 2 ? r.z : r.w;
  const float u = u01(w);
  lv.U[i] = u;
  lv.TH[i] = (float)(lo[j] + (double)u * (hi[j] - lo[j]));
}

// A double's place among the doubles as a whole number (equal for -0 and 0): the
// comparisons below take two integer instructions instead of the FP64 pipe,
// which takes 16 cycles an instruction and warp on this GPU.
__device__ __forceinline__ long long order_key(double x) {
  const long long b = __double_as_longlong(x + 0.0);
  return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

// Ranks of lnL (ascending, ties broken by index) into ord[], one CTA; key: n
// words of scratch.
__device__ void rank_live(int n, const double* lnl_s, long long* key, int* ord) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) key[i] = order_key(lnl_s[i]);
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const long long a = key[i];
    int r = 0;
#pragma unroll 4
    for (int j = 0; j < n; ++j) r += key[j] < a + (j < i);   // b < a, or b == a and j < i
    ord[r] = i;
  }
  __syncthreads();
}

constexpr int SEL_STAGE = 32768;   // bytes: the ranks' keys (8 NSS_MAX_LIVE), then the survivors' coordinates

// Shared memory of k_nss_select in bytes: lnL, step and ln weight of the
// removed points, the stage, ranks, means, and the covariance
size_t sel_smem_bytes(int n, int k, int d, bool full) {
  return 8ull * n + 16ull * k + SEL_STAGE + 4ull * n + 4ull * d + (full ? 4ull * d * d : 0);
}

// One CTA: remove the k lowest live points (evidence, dead records), start the
// chains, and factor the survivors' covariance for the directions.
__global__ void __launch_bounds__(1024) k_nss_select(int n, int k, int d, int iter, Live lv, Dead dd, Chains ch,
                                                     float* chol, NssState* st, uint32_t k0, uint32_t k1) {
  extern __shared__ __align__(16) uint8_t smem[];
  double* lnl_s = reinterpret_cast<double*>(smem);
  double* step_s = lnl_s + n;                 // [k] ln X lost with each removed point
  double* lnw_s = step_s + k;                 // [k] its ln weight
  long long* key = reinterpret_cast<long long*>(lnw_s + k);
  float* stage = reinterpret_cast<float*>(key);
  int* ord = reinterpret_cast<int*>(stage + SEL_STAGE / 4);
  float* mu = reinterpret_cast<float*>(ord + n);
  float* A = mu + d;                          // [d][d] covariance, then its Cholesky factor (full mode)
  __shared__ int s_above, s_nd0;
  __shared__ double red[RED_THREADS / 32];
  const bool full = d <= NSS_FULL_COV;
  const int tid = threadIdx.x;
  for (int i = tid; i < n; i += blockDim.x) lnl_s[i] = lv.lnl[i];
  if (tid == 0) {
    s_above = 0;
    s_nd0 = st->n_dead;
    st->active[0] = st->active[1] = 0;
  }
  // the removed points' shares of the prior volume
  for (int j = tid; j < k; j += blockDim.x) {
    step_s[j] = 1.0 / (double)(n - j);
    lnw_s[j] = log(-expm1(-step_s[j]));
  }
  __syncthreads();
  rank_live(n, lnl_s, key, ord);
  const double lstar = lnl_s[ord[k - 1]];
  int cnt = 0;
  for (int i = tid; i < n; i += blockDim.x) cnt += lnl_s[i] > lstar;
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if ((tid & 31) == 0 && cnt) atomicAdd(&s_above, cnt);
  for (int i = tid; i < n; i += blockDim.x) lv.order[i] = ord[i];
  __syncthreads();
  const int n_above = s_above;
  const int nd0 = s_nd0;
  // dead records: the removed rows, in increasing lnL
  for (int q = tid; q < k * d; q += blockDim.x) {
    const int j = q / d, c = q - j * d;
    if (nd0 + j < dd.cap) dd.TH[(size_t)(nd0 + j) * d + c] = lv.TH[(size_t)ord[j] * d + c];
  }
  if (tid == 0) {
    double lnX = st->lnX;
    for (int j = 0; j < k; ++j) {
      const double step = step_s[j];
      step_s[j] = lnX;
      lnX -= step;
    }
    st->lnX = lnX;
    st->lstar = lstar;
    st->n_above = n_above;
    st->n_dead = nd0 + k;
    if (n_above == 0) st->stop = 2;   // every survivor sits on the contour: nothing left to climb
  }
  __syncthreads();
  for (int j = tid; j < k; j += blockDim.x) {
    const double lnw = step_s[j] + lnw_s[j];
    lnw_s[j] = lnw;
    if (nd0 + j < dd.cap) {
      dd.lnl[nd0 + j] = lnl_s[ord[j]];
      dd.lnw[nd0 + j] = lnw;
    }
  }
  __syncthreads();
  add_points(st, k, [&](int j) { return lnl_s[ord[j]]; }, [&](int j) { return lnw_s[j]; }, red);
  // chains: start at a random survivor strictly above the contour
  for (int c = tid; c < k; c += blockDim.x) {
    const uint4 r = philox(make_uint4((uint32_t)iter, (uint32_t)c, 0u, TAG_START), k0, k1);
    int src = ord[n - 1];
    if (n_above > 0) src = ord[n - n_above + min((int)(u01(r.x) * n_above), n_above - 1)];
    ch.lnl0[c] = lnl_s[src];
    ch.phase[c] = n_above > 0 ? PH_NEW : PH_DONE;
    ch.step[c] = 0; ch.pend[c] = 0; ch.draw[c] = 0;
    ch.nl[c] = 0; ch.nr[c] = 0; ch.ns[c] = 0;
  }
  for (int q = tid; q < k * d; q += blockDim.x) {
    const int c = q / d, j = q - c * d;
    const uint4 r = philox(make_uint4((uint32_t)iter, (uint32_t)c, 0u, TAG_START), k0, k1);
    int src = ord[n - 1];
    if (n_above > 0) src = ord[n - n_above + min((int)(u01(r.x) * n_above), n_above - 1)];
    ch.x0[q] = lv.U[(size_t)src * d + j];
  }
  // covariance of the survivors (all live points but the k removed), unit-cube
  // coordinates.  The survivors pass through shared memory in chunks, loaded by
  // all threads at once; every sum runs over them in order.  (Threads that read
  // the survivors one after the other waited on L2 for each: with that, the
  // evidence and the ranks above in FP64, this kernel took 425 us at 300 points.)
  const int m = n - k, chunk = max(SEL_STAGE / 4 / d, 1);
  const float inv = 1.f / (float)max(m - 1, 1);
  for (int e = tid; e < (full ? d * d : 0); e += blockDim.x) A[e] = 0.f;
  for (int pass = 0; pass < 2; ++pass) {   // means, then covariances or variances
    float s = 0.f;
    for (int q0 = 0; q0 < m; q0 += chunk) {
      const int nq = min(chunk, m - q0);
      if (pass == 0 || m > chunk) {
        __syncthreads();
        for (int e = tid; e < nq * d; e += blockDim.x) {
          const int q = e / d;
          stage[e] = lv.U[(size_t)ord[k + q0 + q] * d + (e - q * d)];
        }
        __syncthreads();
      }
      if (pass == 0) {
        if (tid < d)
          for (int q = 0; q < nq; ++q) s += stage[q * d + tid];
      } else if (!full) {
        if (tid < d)
          for (int q = 0; q < nq; ++q) {
            const float x = stage[q * d + tid] - mu[tid];
            s = fmaf(x, x, s);
          }
      } else {
        for (int e = tid; e < d * d; e += blockDim.x) {
          const int i = e / d, j = e - i * d;
          if (j > i) continue;
          float c = A[e];
          const float mi = mu[i], mj = mu[j];
#pragma unroll 4
          for (int q = 0; q < nq; ++q) c = fmaf(stage[q * d + i] - mi, stage[q * d + j] - mj, c);
          A[e] = c;
        }
      }
    }
    if (tid < d && pass == 0) mu[tid] = s / (float)m;
    if (tid < d && pass == 1 && !full) chol[tid] = sqrtf(s * inv + 1e-14f);
    __syncthreads();
  }
  if (!full) return;
  for (int e = tid; e < d * d; e += blockDim.x) A[e] *= inv;
  __syncthreads();
  for (int j = tid; j < d; j += blockDim.x) mu[j] = A[j * d + j];   // the variances, for the pivot floor
  __syncthreads();
  // right-looking Cholesky in shared memory; a pivot below 1e-7 of its column's
  // variance (a direction the survivors do not span) is raised to that floor
  for (int j = 0; j < d; ++j) {
    if (tid == 0) {
      const float a = A[j * d + j];
      A[j * d + j] = sqrtf(fmaxf(a, 1e-7f * mu[j] + 1e-14f));
    }
    __syncthreads();
    const float pj = A[j * d + j];
    for (int i = j + 1 + tid; i < d; i += blockDim.x) A[i * d + j] /= pj;
    __syncthreads();
    const int rem = d - j - 1;
    for (int e = tid; e < rem * rem; e += blockDim.x) {
      const int i = j + 1 + e / rem, p = j + 1 + e % rem;
      if (p <= i) A[i * d + p] -= A[i * d + j] * A[p * d + j];
    }
    __syncthreads();
  }
  for (int e = tid; e < d * d; e += blockDim.x) {
    const int i = e / d, j = e - i * d;
    chol[e] = j <= i ? A[e] : 0.f;
  }
}

struct RoundArgs {
  int k, d, m_steps, round, iter;
  float w;
  const double *lo, *hi;
  const float* chol;       // [d][d] lower factor (full) or [d] standard deviations
  int full;
  Chains ch;
  const double* lnl_b;     // [k] last round's lnL
  const uint32_t* st_b;    // [k] last round's row status
  float* th_b;             // [k][d] this round's proposals
  NssState* st;
  uint32_t k0, k1;
};

// Columns of the directions' factor kept in shared memory by k_nss_round
constexpr int ROUND_CHOL = 64;
// Shared memory of k_nss_round in bytes: per chain normals, proposal, direction
// and current point, then the factor
size_t round_smem_bytes(int d, bool full) {
  return 4ull * (CHAINS_PER_BLOCK * 4 * d + (full && d <= ROUND_CHOL ? d * d : 0));
}

// One warp per chain: consume the chain's last likelihood, advance its slice
// state machine to its next proposal (proposals outside the unit cube are
// decided without an evaluation) and write it as a parameter row.  The kernel is
// one chain of dependent steps, so what any of them may need (the point, the
// direction, the factor, the prior's box) is loaded at once at its start, and
// the direction is not read back from global memory.
__global__ void __launch_bounds__(CHAINS_PER_BLOCK * 32) k_nss_round(RoundArgs a) {
  sed::pdl_enter();
  extern __shared__ float zsh[];                       // [CHAINS_PER_BLOCK][4][d], then the factor
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c = blockIdx.x * CHAINS_PER_BLOCK + warp;
  if (blockIdx.x == 0 && threadIdx.x == 0) a.st->active[(a.round + 1) & 1] = 0;
  const int d = a.d;
  float* z = zsh + (size_t)warp * 4 * d;
  float* x = z + d;
  float* v = x + d;
  float* x0 = v + d;
  const float* chol = a.chol;
  if (a.full && d <= ROUND_CHOL) {
    float* L = zsh + CHAINS_PER_BLOCK * 4 * d;
    for (int j = threadIdx.x; j < d * d; j += CHAINS_PER_BLOCK * 32) L[j] = a.chol[j];
    chol = L;
  }
  double box_lo = 0.0, box_hi = 0.0;   // the lane's first column
  if (lane < d) { box_lo = a.lo[lane]; box_hi = a.hi[lane]; }
  if (c < a.k)
    for (int j = lane; j < d; j += 32) {
      x0[j] = a.ch.x0[(size_t)c * d + j];
      v[j] = a.ch.v[(size_t)c * d + j];
    }
  __syncthreads();
  if (c >= a.k) return;
  auto write_row = [&](const float* p) {
    for (int j = lane; j < d; j += 32) {
      const double lo = j == lane ? box_lo : a.lo[j], hi = j == lane ? box_hi : a.hi[j];
      a.th_b[(size_t)c * d + j] = (float)(lo + (double)p[j] * (hi - lo));
    }
  };
  bool moved = false, turned = false;   // the point, the direction to be written back
  int ph = a.ch.phase[c], s = a.ch.step[c], nl = a.ch.nl[c], nr = a.ch.nr[c], ns = a.ch.ns[c];
  float tL = a.ch.tL[c], tR = a.ch.tR[c], t = a.ch.t[c];
  uint32_t draw = a.ch.draw[c];
  const double lstar = a.st->lstar;
  bool have = a.ch.pend[c] != 0;
  double lc = have ? a.lnl_b[c] : -INFINITY;
  bool inside = have && a.st_b[c] == 0 && lc > lstar;
  bool wrote = false;
  for (int it = 0; it < 4 * (2 * MAXOUT + MAXSHRINK) && ph != PH_DONE; ++it) {
    if (have) {   // the outcome of the last proposal at t
      have = false;
      if (ph == PH_LEFT) {
        if (inside && nl < MAXOUT) { tL -= a.w; ++nl; } else ph = PH_RIGHT;
      } else if (ph == PH_RIGHT) {
        if (inside && nr < MAXOUT) { tR += a.w; ++nr; } else ph = PH_SHRINK;
      } else if (ph == PH_SHRINK) {
        if (inside) {
          for (int j = lane; j < d; j += 32) x0[j] = fmaf(t, v[j], x0[j]);
          moved = true;
          if (lane == 0) a.ch.lnl0[c] = lc;
          ++s;
          ph = PH_NEW;
        } else {
          if (t < 0.f) tL = t; else tR = t;
          if (++ns >= MAXSHRINK) { ++s; ph = PH_NEW; }
        }
      }
      __syncwarp();
    }
    if (ph == PH_NEW) {
      if (s >= a.m_steps) { ph = PH_DONE; break; }
      // direction: v = L z / |z| with z standard normal (Box-Muller on Philox words)
      float zz = 0.f;
      for (int j0 = 0; j0 < d; j0 += 128) {
        const int j = j0 + 4 * lane;
        if (j < d) {
          const uint4 r = philox(make_uint4((uint32_t)a.iter, (uint32_t)c, draw, TAG_DIR | ((uint32_t)(j >> 2) << 8)),
                                 a.k0, a.k1);
          float s0, c0, s1, c1;
          const float r0 = sqrtf(-2.f * logf(u01(r.x))), r1 = sqrtf(-2.f * logf(u01(r.z)));
          sincospif(2.f * u01(r.y), &s0, &c0);
          sincospif(2.f * u01(r.w), &s1, &c1);
          const float g[4] = {r0 * c0, r0 * s0, r1 * c1, r1 * s1};
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (j + q < d) { z[j + q] = g[q]; zz = fmaf(g[q], g[q], zz); }
        }
      }
      ++draw;
#pragma unroll
      for (int o = 16; o; o >>= 1) zz += __shfl_xor_sync(0xffffffffu, zz, o);
      const float rz = rsqrtf(zz);
      __syncwarp();
      for (int i = lane; i < d; i += 32) {
        float acc = 0.f;
        if (a.full) {
          const float* Li = chol + (size_t)i * d;
          for (int j = 0; j <= i; ++j) acc = fmaf(Li[j], z[j], acc);
        } else {
          acc = chol[i] * z[i];
        }
        v[i] = acc * rz;
      }
      turned = true;
      const uint4 r = philox(make_uint4((uint32_t)a.iter, (uint32_t)c, draw++, TAG_SLICE), a.k0, a.k1);
      tL = -u01(r.x) * a.w;
      tR = tL + a.w;
      nl = nr = ns = 0;
      ph = PH_LEFT;
      __syncwarp();
    }
    if (ph == PH_LEFT) t = tL;
    else if (ph == PH_RIGHT) t = tR;
    else {
      const uint4 r = philox(make_uint4((uint32_t)a.iter, (uint32_t)c, draw++, TAG_SLICE), a.k0, a.k1);
      t = tL + u01(r.x) * (tR - tL);
    }
    bool out = false;
    for (int j = lane; j < d; j += 32) {
      const float xj = fmaf(t, v[j], x0[j]);
      x[j] = xj;
      out |= !(xj >= 0.f && xj <= 1.f);
    }
    out = __any_sync(0xffffffffu, out);
    __syncwarp();
    if (out) {   // outside the box prior: outside the contour, no evaluation
      have = true;
      inside = false;
      continue;
    }
    write_row(x);
    wrote = true;
    break;
  }
  for (int j = lane; j < d; j += 32) {
    if (moved) a.ch.x0[(size_t)c * d + j] = x0[j];
    if (turned) a.ch.v[(size_t)c * d + j] = v[j];
  }
  if (!wrote) write_row(x0);   // an idle row (done chain): evaluated, not used
  if (lane == 0) {
    a.ch.phase[c] = ph; a.ch.step[c] = s; a.ch.nl[c] = nl; a.ch.nr[c] = nr; a.ch.ns[c] = ns;
    a.ch.tL[c] = tL; a.ch.tR[c] = tR; a.ch.t[c] = t; a.ch.draw[c] = draw;
    a.ch.pend[c] = wrote ? 1 : 0;
    if (wrote) atomicAdd(&a.st->n_like, 1ull);
    if (ph != PH_DONE) atomicAdd(&a.st->active[a.round & 1], 1);
  }
}

// One CTA: the chains' end points replace the removed live points; insertion
// ranks among the survivors; the stop test ln(Z_live / Z) < stop_dlnz.
__global__ void __launch_bounds__(1024) k_nss_replace(int n, int k, int d, int iter, const double* lo,
                                                      const double* hi, Live lv, Dead dd, Chains ch, NssState* st,
                                                      double stop_dlnz, int last) {
  __shared__ double red[RED_THREADS / 32];
  __shared__ long long key[NSS_MAX_LIVE];   // the survivors' lnL in order
  const int tid = threadIdx.x;
  const int nd0 = st->n_dead - k;   // first dead record of this iteration
  for (int q = k + tid; q < n; q += blockDim.x) key[q] = order_key(lv.lnl[lv.order[q]]);
  __syncthreads();
  for (int c = tid; c < k; c += blockDim.x) {
    const long long l = order_key(ch.lnl0[c]);
    int q = k, q1 = n;   // they ascend: the first one not below l
    while (q < q1) {
      const int mid = (q + q1) >> 1;
      if (key[mid] < l) q = mid + 1; else q1 = mid;
    }
    if (nd0 + c < dd.cap && dd.rank) dd.rank[nd0 + c] = q - k;
  }
  __syncthreads();
  for (int q = tid; q < k * d; q += blockDim.x) {
    const int c = q / d, j = q - c * d;
    const int slot = lv.order[c];
    const float u = ch.x0[q];
    lv.U[(size_t)slot * d + j] = u;
    lv.TH[(size_t)slot * d + j] = (float)(lo[j] + (double)u * (hi[j] - lo[j]));
  }
  for (int c = tid; c < k; c += blockDim.x) lv.lnl[lv.order[c]] = ch.lnl0[c];
  __syncthreads();
  // ln Z_live = ln X + ln(mean L_live)
  double mx = -INFINITY;
  for (int i = red_start(n); i < n; i += RED_THREADS) mx = fmax(mx, lv.lnl[i]);
  mx = block_reduce<true>(mx, red);
  double sm = 0.0;
  if (mx > -INFINITY)
    for (int i = red_start(n); i < n; i += RED_THREADS) sm += exp(lv.lnl[i] - mx);
  sm = block_reduce<false>(sm, red);
  if (tid == 0) {
    const double lz_live = mx == -INFINITY ? -INFINITY : st->lnX + mx + log(sm) - log((double)n);
    if (st->lnZ > -INFINITY && lz_live - st->lnZ < stop_dlnz) st->stop = 1;
    if (last && !st->stop) st->stop = 3;
  }
}

// One CTA: the final live points join the evidence (weight X / n each, in
// increasing lnL) and the records' weights become ln posterior weights.
__global__ void __launch_bounds__(1024) k_nss_final(int n, int d, Live lv, Dead dd, NssState* st) {
  extern __shared__ __align__(16) uint8_t smem[];
  double* lnl_s = reinterpret_cast<double*>(smem);
  long long* key = reinterpret_cast<long long*>(lnl_s + n);
  int* ord = reinterpret_cast<int*>(key + n);
  __shared__ int s_nd0;
  __shared__ double s_lnw;
  __shared__ double red[RED_THREADS / 32];
  const int tid = threadIdx.x;
  for (int i = tid; i < n; i += blockDim.x) lnl_s[i] = lv.lnl[i];
  if (tid == 0) s_nd0 = st->n_dead;
  __syncthreads();
  rank_live(n, lnl_s, key, ord);
  const int nd0 = s_nd0;
  for (int q = tid; q < n * d; q += blockDim.x) {
    const int j = q / d, c = q - j * d;
    if (nd0 + j < dd.cap) dd.TH[(size_t)(nd0 + j) * d + c] = lv.TH[(size_t)ord[j] * d + c];
  }
  if (tid == 0) s_lnw = st->lnX - log((double)n);
  __syncthreads();
  const double lnw = s_lnw;
  for (int j = tid; j < n; j += blockDim.x)
    if (nd0 + j < dd.cap) {
      dd.lnl[nd0 + j] = lnl_s[ord[j]];
      dd.lnw[nd0 + j] = lnw;
    }
  add_points(st, n, [&](int j) { return lnl_s[ord[j]]; }, [&](int) { return lnw; }, red);
  if (tid == 0) st->n_dead = nd0 + n;
  __syncthreads();
  const double lz = st->lnZ;
  const int nrec = min(st->n_dead, dd.cap);
  for (int i = tid; i < nrec; i += blockDim.x) dd.lnw[i] = dd.lnl[i] + dd.lnw[i] - lz;
}

}  // namespace

extern "C" {

sed_status sed_nss_run(sed_ctx* ctx, sed_model_id model, const sed_nss_desc* desc, float* dead_theta,
                       double* dead_lnl, double* dead_logw, int32_t* ins_rank, int max_dead, sed_nss_result* out,
                       void* stream) {
  if (!ctx || !desc || !out) return SED_EINVAL;
  memset(out, 0, sizeof *out);
  if (model < 0 || model >= (int)ctx->models.size() || !ctx->models[model]) return SED_EINVAL;
  Model* M = ctx->models[model];
  const int d = M->dv.n_param, n = desc->n_live, k = desc->n_replace;
  if (d < 1 || d > NSS_MAX_D) return SED_EINVAL;
  if (n < 2 || n > NSS_MAX_LIVE || k < 1 || k > n / 2 || desc->n_slice_steps < 1 || desc->max_iter < 1)
    return SED_EINVAL;
  if (!desc->lo || !desc->hi || !(desc->stop_dlnz == desc->stop_dlnz) || desc->slice_width < 0.0) return SED_EINVAL;
  for (int j = 0; j < d; ++j)
    if (!(desc->lo[j] < desc->hi[j]) || !isfinite(desc->lo[j]) || !isfinite(desc->hi[j])) return SED_EINVAL;
  if (max_dead < 0) return SED_EINVAL;
  const bool want = dead_theta || dead_lnl || dead_logw || ins_rank;
  const int cap = want ? max_dead : 0;
  const bool full = d <= NSS_FULL_COV;
  int prev = -1;
  cudaGetDevice(&prev);
  cudaSetDevice(ctx->device);
  cudaStream_t s = (cudaStream_t)stream;

  // one device allocation, carved into the run's buffers
  size_t off = 0;
  auto take = [&](size_t bytes) { const size_t o = off; off += (bytes + 255) / 256 * 256; return o; };
  const size_t o_lo = take(8 * d), o_hi = take(8 * d), o_st = take(sizeof(NssState));
  const size_t o_U = take(4ull * n * d), o_TH = take(4ull * n * d), o_lnl = take(8ull * n), o_ord = take(4ull * n);
  const size_t o_x0 = take(4ull * k * d), o_v = take(4ull * k * d), o_l0 = take(8ull * k);
  const size_t o_f = take(4ull * 3 * k), o_i = take(4ull * 7 * k);
  const size_t o_thb = take(4ull * k * d), o_lb = take(8ull * k), o_sb = take(4ull * k);
  const size_t o_ch = take(full ? 4ull * d * d : 4ull * d);
  const size_t o_dth = take(4ull * cap * d), o_dl = take(8ull * cap), o_dw = take(8ull * cap), o_dr = take(4ull * cap);
  const size_t total = off;
  if (!budget_reserve(ctx, total)) {
    cudaSetDevice(prev);
    return SED_ENOMEM;
  }
  uint8_t* base = nullptr;
  if (cudaMalloc(&base, total) != cudaSuccess) {
    budget_release(ctx, total);
    cudaSetDevice(prev);
    return SED_ENOMEM;
  }
  NssState* st_h = nullptr;
  cudaHostAlloc((void**)&st_h, sizeof(NssState), cudaHostAllocDefault);
  sed_status ret = SED_OK;
  auto F = [&](size_t o) { return base + o; };
  double* lo_d = (double*)F(o_lo);
  double* hi_d = (double*)F(o_hi);
  NssState* st = (NssState*)F(o_st);
  Live lv{(float*)F(o_U), (float*)F(o_TH), (double*)F(o_lnl), (int*)F(o_ord)};
  Chains ch{};
  ch.x0 = (float*)F(o_x0); ch.v = (float*)F(o_v); ch.lnl0 = (double*)F(o_l0);
  float* fb = (float*)F(o_f);
  ch.tL = fb; ch.tR = fb + k; ch.t = fb + 2 * k;
  int* ib = (int*)F(o_i);
  ch.phase = ib; ch.step = ib + k; ch.nl = ib + 2 * k; ch.nr = ib + 3 * k; ch.ns = ib + 4 * k; ch.pend = ib + 5 * k;
  ch.draw = (uint32_t*)(ib + 6 * k);
  float* th_b = (float*)F(o_thb);
  double* lnl_b = (double*)F(o_lb);
  uint32_t* st_b = (uint32_t*)F(o_sb);
  float* chol = (float*)F(o_ch);
  Dead dd{(float*)F(o_dth), (double*)F(o_dl), (double*)F(o_dw), (int*)F(o_dr), cap};
  const uint32_t k0 = (uint32_t)desc->seed, k1 = (uint32_t)(desc->seed >> 32);
  const float w = desc->slice_width > 0.0 ? (float)desc->slice_width : sqrtf((float)d + 2.f);
  const size_t sel_smem = sel_smem_bytes(n, k, d, full);
  const size_t fin_smem = 20ull * n;
  const size_t round_smem = round_smem_bytes(d, full);
  static DynSmemCache a_sel, a_fin, a_round;
  const long long max_rounds = (long long)desc->n_slice_steps * (2 * MAXOUT + MAXSHRINK) + 4;
  long long n_rows = n;
  int iter = 0;
  auto CKE = [&](cudaError_t e) {
    if (e != cudaSuccess && !ret) {
      ctx->last_error = std::string("nss: ") + cudaGetErrorString(e);
      ret = SED_ECUDA;
    }
    return e == cudaSuccess;
  };
  CKE(cudaMemcpyAsync(lo_d, desc->lo, 8 * d, cudaMemcpyHostToDevice, s));
  CKE(cudaMemcpyAsync(hi_d, desc->hi, 8 * d, cudaMemcpyHostToDevice, s));
  CKE(cudaMemsetAsync(ib, 0, 4ull * 7 * k, s));
  CKE(ensure_dyn_smem(k_nss_select, sel_smem, &a_sel));
  CKE(ensure_dyn_smem(k_nss_final, fin_smem, &a_fin));
  CKE(ensure_dyn_smem(k_nss_round, round_smem, &a_round));
  if (!ret) {
    k_nss_init<<<(n * d + 255) / 256, 256, 0, s>>>(n, d, lo_d, hi_d, lv, st, k0, k1);
    CKE(cudaGetLastError());
  }
  if (!ret) ret = sed_loglike(ctx, model, lv.TH, n, d, lv.lnl, nullptr, desc->precision, stream);
  for (; !ret && iter < desc->max_iter; ++iter) {
    k_nss_select<<<1, 1024, sel_smem, s>>>(n, k, d, iter, lv, dd, ch, chol, st, k0, k1);
    if (!CKE(cudaGetLastError())) break;
    RoundArgs ra{};
    ra.k = k; ra.d = d; ra.m_steps = desc->n_slice_steps; ra.iter = iter; ra.w = w;
    ra.lo = lo_d; ra.hi = hi_d; ra.chol = chol; ra.full = full; ra.ch = ch;
    ra.lnl_b = lnl_b; ra.st_b = st_b; ra.th_b = th_b; ra.st = st; ra.k0 = k0; ra.k1 = k1;
    long long r = 0;
    bool done = false;
    while (!done && !ret) {
      for (int q = 0; q < ROUNDS && !ret; ++q, ++r) {
        ra.round = (int)(r & 1);
        if (!CKE(sed::launch_pdl(k_nss_round, dim3((k + CHAINS_PER_BLOCK - 1) / CHAINS_PER_BLOCK),
                                 dim3(CHAINS_PER_BLOCK * 32), round_smem, s, ra))) break;
        ret = sed_loglike(ctx, model, th_b, k, d, lnl_b, st_b, desc->precision, stream);
        n_rows += k;
      }
      if (ret) break;
      CKE(cudaMemcpyAsync(st_h, st, sizeof(NssState), cudaMemcpyDeviceToHost, s));
      CKE(cudaStreamSynchronize(s));
      if (ret) break;
      done = st_h->active[(int)((r - 1) & 1)] == 0;
      if (!done && r > max_rounds) {
        ctx->last_error = "nss: slice chains did not finish";
        ret = SED_ECUDA;
      }
    }
    if (ret) break;
    k_nss_replace<<<1, 1024, 0, s>>>(n, k, d, iter, lo_d, hi_d, lv, dd, ch, st, desc->stop_dlnz,
                                     iter + 1 == desc->max_iter);
    CKE(cudaGetLastError());
    CKE(cudaMemcpyAsync(st_h, st, sizeof(NssState), cudaMemcpyDeviceToHost, s));
    CKE(cudaStreamSynchronize(s));
    if (!ret && st_h->stop) {
      ++iter;
      break;
    }
  }
  if (!ret) {
    k_nss_final<<<1, 1024, fin_smem, s>>>(n, d, lv, dd, st);
    CKE(cudaGetLastError());
    CKE(cudaMemcpyAsync(st_h, st, sizeof(NssState), cudaMemcpyDeviceToHost, s));
    CKE(cudaStreamSynchronize(s));
  }
  if (!ret) {
    out->lnz = st_h->lnZ;
    out->info_h = st_h->H;
    out->n_iter = iter;
    out->n_dead = st_h->n_dead;
    out->converged = st_h->stop == 1 || st_h->stop == 2;
    out->n_like = (int64_t)st_h->n_like;
    out->n_rows = n_rows;
    const int nrec = std::min(st_h->n_dead, cap);
    if (dead_theta) CKE(cudaMemcpy(dead_theta, dd.TH, 4ull * nrec * d, cudaMemcpyDeviceToHost));
    if (dead_lnl) CKE(cudaMemcpy(dead_lnl, dd.lnl, 8ull * nrec, cudaMemcpyDeviceToHost));
    if (dead_logw) CKE(cudaMemcpy(dead_logw, dd.lnw, 8ull * nrec, cudaMemcpyDeviceToHost));
    if (ins_rank) CKE(cudaMemcpy(ins_rank, dd.rank, 4ull * std::min(nrec, iter * k), cudaMemcpyDeviceToHost));
    if (!ret && want && st_h->n_dead > cap) {
      ctx->last_error = "nss: max_dead below the points of the run";
      ret = SED_ERANGE;
    }
  }
  cudaStreamSynchronize(s);
  cudaFree(base);
  budget_release(ctx, total);
  if (st_h) cudaFreeHost(st_h);
  cudaSetDevice(prev);
  return ret;
}

}  // extern "C"
