// Fused epilogue: attenuation + nebular, observer-frame scaling, photometric
// and spectral projections and the Gaussian log-likelihood.  One CTA per
// parameter row; the attenuated rest-frame spectrum of the row is staged in
// shared memory once and every projection gathers from it.
//
//  F(lam) = e^{-tau_d(lam)} [ e^{-tau_BC(lam)} (Y(lam) + neb(lam)) + O(lam) ]
//     tau_BC = tau_pow (lam/5500)^alpha_pow (birth cloud, Sec. 2.4)
//     tau_d  = diffuse power law, or Kriek & Conroy 2013 (Sec. 2.4)
//     neb    = Q_young 10^(bilinear log10 template)        (App. C)
//  photometry (App. D, Eq. app_phot_T): m_b = P sum_j w_j lerp(F/lam^2)(lam_j/(1+z))
//  spectrum (App. E, Eq. app_response): m_i = s sum_j w_ij F_j / sum_j w_ij,
//     Gaussian in ln(lam) truncated at 5 sigma, linear interpolation for
//     kernels narrower than half a model log-pixel
//  lnL (Eq. total_lnlike): sum over included data of -r^2/2 - ln(2 pi sigma^2)/2
//     (r = (d - m)/sigma, min(r, 0) for a band that is an upper limit, Eq.
//     app_line_chi2_UL), with sigma_eff for sigma under the optional noise
//     floor (App. sys_floor) and the marginalised calibration polynomial's
//     terms (App. E); spectral residuals in FP32 on the host's d/sigma and
//     1/sigma, the bands' terms and every sum across threads in FP64
//  emission lines (App. C, App. line_proj): F_l = Q_young 10^(bilinear log10
//     cube) x the nebular attenuation at lam_l x s / (1+z); photometry
//     + F_l R_b(lam_obs) lam_obs / Z_b; spectrum + F_l (lam_i/c) N(ln lam_i;
//     ln lam_obs, s_l), s_l = sqrt(sigma_gas^2 + sigma_inst^2(lam_obs))/c
//     (Eq. app_line_profile); line catalogue: blends of F_l, one-sided upper
//     limits (Eq. app_line_chi2_det, Eq. app_line_chi2_UL)
//
// All reductions run in a fixed order, so the result is bitwise reproducible.
#include "sed_internal.cuh"
#include "locate.cuh"
#include "atten.cuh"
#include "calib.cuh"
#include "floor.cuh"
#include "igm.cuh"
#include "lines.cuh"

namespace sed {

// 128 threads per row and a small shared-memory window keep every row of a
// paper-scale batch resident at once (7 CTAs per SM, 1064 rows on 152 SMs):
// the kernel is bound by the latency of its gathers, so rows in flight is what
// sets its speed, and the 72 registers that 7 CTAs leave a thread (against 64
// at 8) keep more of each thread's loads in flight (measured 0.0988 against
// 0.1029 ms per 1024-row step).  Of a 1024-row photometric launch the row's
// fixed part takes about 6 us, its nodes 11 us and its samples 6 us; copying Y
// and O of all nodes at once, one load for the nebular corners, samples without
// walks and shared-memory words without the pairs' bank conflicts took the
// epilogue stage from 34.8 to 26.6 us (1024 rows) and 116.7 to 79.9 us (4096
// rows, BF16).
constexpr int EPI_THREADS = 128;
constexpr int EPI_WARPS = EPI_THREADS / 32;
constexpr int MAX_BANDS = 128;

// A launch that leaves most of the chip's warps empty takes 256 or 512 threads
// per row (NT): a row is one chain of dependent loads, and spreading its
// nodes, filter samples and pixels over more warps shortens the chain (64 rows
// of the paper-scale photometric fit: epilogue stage 28.7 -> 16.4 us, step 54.1 ->
// 37.7 us; 301 rows with a 1111-pixel spectrum: 59.4 -> 28.7 us).  Every sum keeps the
// 128-thread instance's terms and order, so a row's result does not depend on
// the instance that computed it: the samples' interpolated values go through
// shared memory where they are spread over all threads, the pixels' residuals
// always do, and the sums over them run as lanes of a warp per band and as
// EPI_THREADS threads over the pixels.  EPI_MISSED marks an excluded pixel there
// (a NaN no arithmetic produces).
constexpr uint32_t EPI_MISSED = 0x7fa00001u;
// From this many threads on, a band's samples are spread over all of them; below
// it a warp takes a band (no shared memory for the samples' values, which would
// cost the 256-thread instance with a spectrum its fourth CTA per SM).
constexpr int EPI_FLAT = 512;

// dynamic shared memory: lam, F/lam^2 and F over the row's window, the
// included pixels' mu/sigma for the calibration moments, with emission lines,
// per line ln(lam_obs) (an FP32 pair), F_l, A_l and 1/s_l, from EPI_FLAT threads on
// the samples' values, and the bands' extents and data where there is room for
// them (a window of some 19,000 nodes with a spectrum leaves none).  The pixels'
// residuals pass through lam's and F/lam^2's places, which the spectrum does not
// read, as many pixels at a time as fit there: no number of pixels needs more.
size_t epilogue_lines_off(const EpiArgs& a) {   // in floats, even (float2 alignment)
  const int np = a.row_model ? a.smem_pix : a.md.n_pix;
  const size_t W = (size_t)(a.row_model ? a.smem_win : a.md.win_max);
  const bool calib = a.row_model || a.md.calib_n > 0;
  const size_t f = 2 * W + (np > 0 ? W : 0) + (calib ? (size_t)np : 0);
  return (f + 1) & ~(size_t)1;
}
size_t epilogue_samp_off(const EpiArgs& a) {   // in floats
  const bool lines = a.row_model ? a.g.n_line > 0 : a.md.use_lines != 0;
  return epilogue_lines_off(a) + (lines ? (size_t)5 * a.g.n_line : 0);
}
size_t epilogue_samp_end(const EpiArgs& a, int nt) {   // in floats
  return epilogue_samp_off(a) + (nt >= EPI_FLAT ? 32 * (size_t)(a.row_model ? a.smem_samp : a.md.n_samp32) : 0);
}
size_t epilogue_band_off(const EpiArgs& a, int nt) {   // in floats, even (double alignment)
  return (epilogue_samp_end(a, nt) + 1) & ~(size_t)1;
}
size_t epilogue_smem(const EpiArgs& a, int nt, bool bands) {
  if (!bands) return epilogue_samp_end(a, nt) * sizeof(float);
  const size_t nb = a.row_model ? MAX_BANDS : a.md.n_filt;
  return epilogue_band_off(a, nt) * sizeof(float) + nb * sizeof(double3) + (nb + 1) * sizeof(int);
}

// a / b by the hardware's reciprocal, subnormals as zero (a and b here are
// differences of wavelengths: zero or far above the subnormals)
__device__ __forceinline__ float div_approx(float a, float b) {
  float q;
  asm("div.approx.ftz.f32 %0, %1, %2;" : "=f"(q) : "f"(a), "f"(b));
  return q;
}

// MULTI: rows of several fits (serving), row r reads model mtab[row_model[r]];
// otherwise every row reads the model in the kernel parameters.  LINES: an
// instance with the emission lines (the one without keeps its code free of them).
// VAR: 1 the age-binned attenuation (one Y per attenuated block), 2 the
// nebular age axis (per-age ionising weights); 0 neither.
template <bool MULTI, bool LINES, int VAR, int NT>
__global__ void __launch_bounds__(NT, NT == EPI_THREADS ? 7 : 1024 / NT) k_epilogue(const __grid_constant__ EpiArgs a) {
  const int r = blockIdx.x;
  if constexpr (MULTI) pdl_enter();
  const ModelDev& md = MULTI ? a.mtab[a.row_model[a.rs[r].orig]] : a.md;
  const GridDev& g = a.g;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int N = g.n_lam;
  // shared memory holds the row's node window [k_lo, k_hi] only (at most
  // md.win_max nodes); the pointers below are offset so that they are indexed
  // by the global node k
  extern __shared__ float4 smem4[];
  const int WIN = MULTI ? a.smem_win : md.win_max;
  __shared__ float mb_s[MAX_BANDS];
  __shared__ double red[EPI_WARPS];
  __shared__ float cal_part[EPI_WARPS][CAL_NV];    // per-warp calibration sums
  __shared__ float cal_L[SED_MAX_CALIB * SED_MAX_CALIB], cal_D[SED_MAX_CALIB], cal_c[SED_MAX_CALIB];  // M = L L^T, 1/L_ii, c*
  __shared__ double cal_fix;                       // the row's lnL terms that do not sum over pixels

  // the bands' extents and data, read in the shadow of the kernel before
  double3* band_s = reinterpret_cast<double3*>(reinterpret_cast<float*>(smem4) + a.band_off);
  int* b32_s = reinterpret_cast<int*>(band_s + (MULTI ? MAX_BANDS : md.n_filt));
  auto band_data = [&](int b) { return make_double3(md.phot_d[b], md.phot_isig[b], md.phot_nlog[b]); };
  auto band = [&](int b) { return a.band_off ? band_s[b] : band_data(b); };   // {datum, 1/sigma, -ln(2 pi sigma^2)/2}
  auto b32 = [&](int b) { return a.band_off ? b32_s[b] : __ldg(md.band32 + b); };
  for (int b = tid; a.band_off && b <= md.n_filt && md.n_filt > 0; b += NT) {
    b32_s[b] = md.band32[b];
    if (b < md.n_filt) band_s[b] = band_data(b);
  }
  if constexpr (!MULTI) pdl_enter();

  if (a.win_reset && r == 0) empty_windows(a.win_reset, a.win_mt);
  if (a.mask_reset && r == 0)
    for (int i = tid; i < a.mask_words; i += NT) a.mask_reset[i] = 0u;
  RowScal rs = a.rs[r];
  if (a.err && *a.err) rs.status |= SED_ROW_DEVICE_TIMEOUT;
  const int ro = rs.orig;   // the caller's row index
  if (rs.status) {
    for (int b = tid; b < md.n_filt; b += blockDim.x)
      if (a.phot_out) a.phot_out[(size_t)ro * md.n_filt + b] = 0.f;
    for (int i = tid; i < md.n_pix; i += blockDim.x)
      if (a.spec_out) a.spec_out[(size_t)ro * md.n_pix + i] = 0.f;
    if (LINES && a.lines_out)
      for (int l = tid; l < g.n_line; l += blockDim.x) a.lines_out[(size_t)ro * g.n_line + l] = 0.f;
    if (tid == 0) {
      if (a.lnl) a.lnl[ro] = -INFINITY;
      if (a.status) a.status[ro] = rs.status;
    }
    return;
  }

  // ---- attenuated rest-frame spectrum of the row's node window into shared memory
  const float* Yr = a.Y + (size_t)r * a.ldn;
  const float* Or = a.O + (size_t)r * a.ldn;
  const float* O2r = a.O2 && a.split && *a.split ? a.O2 + (size_t)r * a.ldn : nullptr;
  const float eb = 0.85f - 1.9f * rs.delta;
  const float opz = 1.f / rs.inv1pz;
  // nebular age axis: the row's Q-weighted weight of each nebular SSP age
  __shared__ float qa_s[MAX_NEB_AGE];
  const float* qa = nullptr;
  if constexpr (VAR == 2) {
    for (int i = tid; i < g.neb_na; i += blockDim.x) qa_s[i] = a.qneb[(size_t)r * MAX_NEB_AGE + i];
    __syncthreads();
    qa = qa_s;
  }
  const bool spec = md.n_pix > 0;
  const int k_lo = rs.k_lo, k_hi = min(rs.k_hi, rs.k_lo + WIN - 1);   // nodes [k_lo, k_hi] are the only ones read below
  // Rest-frame lambda and F / lam^2, as two arrays: a warp's samples lie one to
  // two nodes apart, so one word per node makes half the bank conflicts of a pair
  float* Ls = reinterpret_cast<float*>(smem4) - k_lo;
  float* Gs = Ls + WIN;
  float* Fs = Gs + WIN;                                                // F (spectral arm only)
  float* mu_s = reinterpret_cast<float*>(smem4) + 3 * WIN;             // calibration: included pixels' mu/sigma (0 elsewhere)
  // Y and O of all the thread's nodes are copied to the nodes' own places in the
  // two arrays at once; the other loads of the next node are issued before this
  // node's arithmetic (the loop, not unrolled, waits on L2 otherwise)
  if constexpr (VAR != 1)
    for (int k = k_lo + tid; k <= k_hi; k += NT) {
      cp_async4(Ls + k, Yr + k);
      cp_async4(Gs + k, Or + k);
    }
  struct Node { float o2; float4 c, nt; };
  auto load_node = [&](int k, Node& v) {
    if (k > k_hi) return;
    v.c = __ldg(g.att4 + k);
    v.o2 = VAR == 1 ? Or[k] : O2r ? O2r[k] : 0.f;
    if (VAR == 1 && O2r) v.o2 = v.o2 + O2r[k];
    if (VAR == 0 && md.use_neb) v.nt = neb_corners(rs, g, k);
  };
  Node nx{};
  load_node(k_lo + tid, nx);
  cp_async_wait_all();
#pragma unroll 1
  for (int k = k_lo + tid; k <= k_hi; k += NT) {
    const Node v = nx;
    load_node(k + NT, nx);
    const float4 c = v.c;
    const float ys = a.lam8 ? rs.y_scale * a.lam8[k] : 1.f;
    float F;
    if constexpr (VAR == 1) {
      float yv[MAX_SEG];
#pragma unroll
      for (int sg = 0; sg < MAX_SEG; ++sg) yv[sg] = sg < md.n_seg ? Yr[sg * a.seg_stride + k] * ys : 0.f;
      F = attenuated_bins(md, rs, c, eb, yv, v.o2 * ys, g, k);
    } else {
      const float o = O2r ? Gs[k] + v.o2 : Gs[k];
      const float nb = !md.use_neb ? 0.f : VAR == 2 ? neb_emission(rs, g, qa, k) : neb_emission(rs, v.nt);
      F = attenuated(md, rs, c, eb, Ls[k] * ys, o * ys, nb, k);
    }
    if (md.use_igm && c.w < IGM_LYA) {   // the IGM transmission at the node's observed wavelength
      float tau, dtau;
      igm_madau(c.w, opz, tau, dtau);
      F *= __expf(-rs.igm_f * tau);
    }
    if (spec) Fs[k] = F;
    Ls[k] = c.w;
    Gs[k] = __fdividef(F, c.w * c.w);
  }
  // emission lines: ln(lam_obs) pairs, fluxes F_l, profile peaks A_l = F_l /
  // (sqrt(2 pi) s_l) and 1/s_l in the tail of the dynamic shared memory
  const int NLn = LINES && md.use_lines ? g.n_line : 0;
  float2* ln_x = reinterpret_cast<float2*>(reinterpret_cast<float*>(smem4) + a.lines_off);
  float* ln_F = reinterpret_cast<float*>(ln_x + NLn);
  float* ln_A = ln_F + NLn;
  float* ln_is = ln_A + NLn;
  for (int l = tid; l < NLn; l += NT) line_setup(md, g, rs, eb, l, ln_F, ln_A, ln_is, ln_x);
  __syncthreads();
  if (LINES && a.lines_out) {   // the lines' fluxes only (sed_line_fluxes)
    for (int l = tid; l < NLn; l += NT) a.lines_out[(size_t)ro * NLn + l] = ln_F[l];
    if (!a.lnl && !a.phot_out && !a.spec_out) return;
  }

  // ---- photometry.  Each sample's bracket starts from the index table over
  //      ln(lambda) at its rest-frame wavelength and is corrected within the
  //      row's window in shared memory; any start gives the same bracket.
  const float lam0 = g.lam_f[0], lamN = g.lam_f[N - 1];
  const int kmin = k_lo, kmax = k_hi - 1;
  // A table cell is half the smallest node spacing wide, and a sample's place in
  // it carries an error below 8e-6 in ln(lambda) (lg2's 2^-22 of its value,
  // 2.6e-6, and the roundings of ln lambda, 1/h and the place, 2.1e-6 together): with that
  // taken off the place, the table's node is the bracket or the one before it as
  // long as the slack stays below a quarter of a cell.  With every sample inside
  // the grid (the window then holds all the nodes) such a sample needs no walk and
  // no clamping but at the grid's end: it tests the next node and takes its
  // bracket, so that a lane's samples run side by side.  The phase is bound by
  // the wavefronts of its loads (the samples, the table, two words of each
  // bracket node), not by arithmetic.
  const float slack = 8e-6f * g.lut_inv_h;
  const bool pick = slack <= 0.25f && k_hi - k_lo >= 2 && md.samp_lam_min * rs.inv1pz >= lam0 &&
                    md.samp_lam_max * rs.inv1pz <= lamN;
  const float q_mul = 0.6931471805599453f * g.lut_inv_h, q_add = fmaf(-g.lut_x0, g.lut_inv_h, -slack);
  auto lerp_at = [&](float x, float l0, float l1, float g0, float g1) {
    const float t = div_approx(x - l0, l1 - l0);
    return g0 + t * (g1 - g0);
  };
  // place in the table, and F/lam^2, at the rest-frame wavelength x
  auto sample_start = [&](float x) { return (int)__ldg(g.lut + (int)fmaf(lg2_approx(x), q_mul, q_add)); };
  auto sample_pick = [&](float x, int k) {
    k = min(k, kmax - 1);
    const float l1 = Ls[k + 1];
    const bool up = l1 <= x;
    const float lx = Ls[up ? k + 2 : k];
    const float* G = Gs + (up ? k + 1 : k);
    return lerp_at(x, up ? l1 : lx, up ? lx : l1, G[0], G[1]);
  };
  auto sample_walk = [&](float x) {
    if (!(x >= lam0 && x <= lamN)) return 0.f;
    int kc = g.lut[min(max((int)fmaf(lg2_approx(x), q_mul, q_add), 0), g.lut_n - 1)];
    kc = min(max(kc, kmin), kmax);
#pragma unroll 1
    while (kc < kmax && Ls[kc + 1] <= x) ++kc;
#pragma unroll 1
    while (kc > kmin && Ls[kc] > x) --kc;
    return lerp_at(x, Ls[kc], Ls[kc + 1], Gs[kc], Gs[kc + 1]);
  };
  // the band's flux from its lanes' sample sums, plus the lines in it (one line
  // per lane); a fixed shuffle tree keeps the order of the sum fixed
  auto band_finish = [&](int b, float acc) {
#pragma unroll
    for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    float lsum = 0.f;
    if (LINES && NLn) {
      for (int l = lane; l < NLn; l += 32) lsum += line_in_band(md, g, rs, b, l, ln_F[l]);
#pragma unroll
      for (int o = 16; o; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    }
    if (lane == 0) {
      const float mb = LINES && NLn ? fmaf(rs.p_phot, acc, lsum) : rs.p_phot * acc;
      if (a.phot_out) a.phot_out[(size_t)ro * md.n_filt + b] = mb;
      mb_s[b] = mb;
    }
  };
  float* rn_s = reinterpret_cast<float*>(smem4);                // the pixels' residuals, 2 WIN at a time
  float* v_s = reinterpret_cast<float*>(smem4) + a.samp_off;    // NT >= EPI_FLAT: the samples' values
  if constexpr (NT < EPI_FLAT) {
    // one band per warp: consecutive lanes take consecutive samples (coalesced
    // loads, eight in flight per lane); a sample outside the grid adds zero
    for (int b = warp; b < md.n_filt; b += NT / 32) {
      float acc = 0.f;
      const int s0 = b32(b);
      const float2* s2 = md.samp32 + 32 * s0 + lane;
      for (int n32 = b32(b + 1) - s0; n32 > 0; n32 -= 8, s2 += 256) {
        if (pick) {
          float2 sp[8];
          int kg[8];
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (u < n32) sp[u] = __ldg(s2 + 32 * u);
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (u < n32) {
              sp[u].x *= rs.inv1pz;
              kg[u] = sample_start(sp[u].x);
            }
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (u < n32) acc = fmaf(sp[u].y, sample_pick(sp[u].x, kg[u]), acc);
        } else {
#pragma unroll 1
          for (int u = 0; u < min(n32, 8); ++u) {
            const float2 sp = __ldg(s2 + 32 * u);
            acc = fmaf(sp.y, sample_walk(sp.x * rs.inv1pz), acc);
          }
        }
      }
      band_finish(b, acc);
    }
  } else {
    const int ns = 32 * md.n_samp32;
    if (pick) {
      for (int j0 = tid; j0 < ns; j0 += 4 * NT) {
        float x[4];
        int kg[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (j0 + u * NT < ns) x[u] = __ldg(&md.samp32[j0 + u * NT].x) * rs.inv1pz;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (j0 + u * NT < ns) kg[u] = sample_start(x[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (j0 + u * NT < ns) v_s[j0 + u * NT] = sample_pick(x[u], kg[u]);
      }
    } else {
#pragma unroll 1
      for (int j = tid; j < ns; j += NT) v_s[j] = sample_walk(__ldg(&md.samp32[j].x) * rs.inv1pz);
    }
  }

  if constexpr (NT >= EPI_FLAT) {
    __syncthreads();
    for (int b = warp; b < md.n_filt; b += NT / 32) {
      float acc = 0.f;
      const int j1 = 32 * b32(b + 1);
#pragma unroll 8
      for (int j = 32 * b32(b) + lane; j < j1; j += 32) acc = fmaf(__ldg(&md.samp32[j].y), v_s[j], acc);
      band_finish(b, acc);
    }
  }

  // ---- spectrum: two neighbouring pixels per thread, which share most of their
  //      nodes, so that a node's position and flux are loaded once for both.  (The
  //      loop over the nodes is bound by instruction issue: 12.5 per pixel and
  //      node against 23 with one pixel per thread.  Epilogue stage of 1024 rows of
  //      1500 pixels with 30 lines 104.5 -> 79.9 us, of 512 calibrated rows 65.5 ->
  //      53.2 us.)  Per-pixel terms in FP32 on
  //      the normalised residual (d - mu)/sigma; the constants
  //      -1/2 ln(2 pi sigma^2) in FP64.
  double part = 0.0;
  float chi = 0.f;
  for (int c0 = 0; c0 < md.n_pix; c0 += 2 * WIN) {   // pixels [c0, last]
    __syncthreads();   // lam and F/lam^2, or the residuals before these, have been read
    const float ll0 = g.lnl_hi[0], llN = g.lnl_hi[N - 1];
    const int last = min(c0 + 2 * WIN, md.n_pix) - 1;
    for (int ib = c0 + 2 * 32 * warp; ib <= last; ib += 2 * NT) {
      float2 pl[2];
      float v[2], xh[2], xl[2], inv_s[2], sw[2] = {0.f, 0.f}, sf[2] = {0.f, 0.f};
      bool gauss[2], valid[2];
      int jl = k_hi, jh = k_lo - 1;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int i = min(ib + 2 * lane + q, last);
        pl[q] = md.pix_ln2[i];
        ln_rest(pl[q], rs.ln1pz_hi, rs.ln1pz_lo, xh[q], xl[q]);
        v[q] = 0.f;
        valid[q] = gauss[q] = false;
        inv_s[q] = 0.f;
        if (xh[q] >= ll0 && xh[q] <= llN) {
          // total dispersion: fixed, or sigma_fix composed with the row's sigma_gal (Eq. one_kernel)
          const float s = md.sample_sgal ? sqrtf(md.pix_fix2[i] + rs.sg_ln * rs.sg_ln) : md.pix_s[i];
          const int k = locate_ln(g, xh[q], g.lnl_hi);
          const float2 n0 = __ldg(g.lnl2 + k), n1 = __ldg(g.lnl2 + k + 1);
          const float dln = (n1.x - n0.x) + (n1.y - n0.y);
          if (s < 0.5f * dln) {
            const float t = ((xh[q] - n0.x) + (xl[q] - n0.y)) / dln;
            v[q] = Fs[k] + t * (Fs[k + 1] - Fs[k]);
            valid[q] = true;
          } else {
            // the nodes within 5 dispersions: a superset of them from the index
            // table alone (each entry within one node of the exact bracket; the
            // margins cover that), clamped to the row's window, which holds every
            // node within 5 dispersions of a pixel; a node past 5 dispersions is
            // left out by predication, so the loop carries no branch (its loads
            // pipeline)
            gauss[q] = true;
            inv_s[q] = 1.f / s;
            int qa = (int)((fmaxf(xh[q] - 5.f * s, ll0) - g.lut_x0) * g.lut_inv_h);
            int qb = (int)((fminf(xh[q] + 5.f * s, llN) - g.lut_x0) * g.lut_inv_h);
            qa = min(max(qa, 0), g.lut_n - 1);
            qb = min(max(qb, 0), g.lut_n - 1);
            jl = min(jl, max(g.lut[qa] - 1, k_lo));
            jh = max(jh, min(g.lut[qb] + 3, k_hi));
          }
        }
      }
#pragma unroll 4
      for (int j = jl; j <= jh; ++j) {
        const float2 n = __ldg(g.lnl2 + j);
        const float f = Fs[j];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const float u = ((n.x - xh[q]) + (n.y - xl[q])) * inv_s[q];
          const float u2 = u * u, w = gauss_w(u2);
          if (u2 <= 25.f) {   // predicated: a node past 5 dispersions is left out
            sw[q] += w;
            sf[q] = fmaf(w, f, sf[q]);
          }
        }
      }
      float la[2] = {0.f, 0.f};
      if (LINES && NLn)
        lines_at_pixels(NLn, ln_A, ln_is, ln_x, pl[0], pl[1], __shfl_sync(0xffffffffu, pl[0].x, 0),
                        __shfl_sync(0xffffffffu, pl[1].x, 31), lane, la[0], la[1]);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int i = ib + 2 * lane + q;
        if (i > last) break;
        if (gauss[q] && sw[q] > 0.f) { v[q] = sf[q] / sw[q]; valid[q] = true; }
        const float mi = LINES && NLn ? fmaf(rs.s_spec, v[q], la[q] * md.pix_lamc[i]) : rs.s_spec * v[q];
        if (a.spec_out) a.spec_out[(size_t)ro * md.n_pix + i] = mi;
        const float isf = md.spec_isf[i];
        const bool inc = valid[q] && isf != 0.f;
        const float ms = inc ? mi * isf : 0.f;   // mu / sigma
        const float dn = md.spec_dn[i];
        float t = dn - ms;                       // (d - mu) / sigma
        if (inc && md.floor_bits[1]) {           // sigma_eff of Eq. app_noise_floor
          const float qf = floor_q(rs.fl[1], ms, dn, rs.fl[1][3] * isf);
          t = t * t / qf + logf(qf);
        }
        rn_s[i - c0] = inc ? t : __uint_as_float(EPI_MISSED);
        if (md.calib_n) mu_s[i] = ms;
      }
    }
    __syncthreads();
    if (NT == EPI_THREADS || tid < EPI_THREADS)
      for (int i = c0 + ((tid - c0) & (EPI_THREADS - 1)); i <= last; i += EPI_THREADS) {   // the pixels tid, tid + 128, ...
        // an included pixel's term: the residual squared, or twice minus the term
        // with the noise floor
        const float t = rn_s[i - c0];
        if (__float_as_uint(t) == EPI_MISSED) continue;
        if (md.floor_bits[1]) chi -= 0.5f * t;
        else chi = fmaf(-0.5f * t, t, chi);
        part += md.spec_nlog[i];
      }
  }
  // the first EPI_WARPS warps own the pixels in every instance; without pixels
  // there is nothing to sum (the FP64 pipe serves the whole SM)
  const bool own = md.n_pix > 0 && (NT == EPI_THREADS || tid < EPI_THREADS);
  if (own) part += (double)chi;
  // calibration moments over each thread's pixels in three blocks of sums
  // (S_0..12, S_13..24, b_0..12), each summed per warp
  if (md.calib_n && own) {
    calib_block<0, 0, EPI_THREADS>(md, mu_s, cal_c, tid, lane, warp, &cal_part[0][0]);
    calib_block<SED_MAX_CALIB, 0, EPI_THREADS>(md, mu_s, cal_c, tid, lane, warp, &cal_part[0][0]);
    calib_block<0, 1, EPI_THREADS>(md, mu_s, cal_c, tid, lane, warp, &cal_part[0][0]);
  }
  if (own) {
#pragma unroll
    for (int o = 16; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if (lane == 0) red[warp] = part;
  }
  __syncthreads();
  if (md.calib_n) {
    // sum the warps' moments in warp order into row 0, factor M and solve for
    // c*; refine c* once from the pixels' calibrated residuals; then each
    // included pixel's change of its term under the polynomial p = A c*
    if (warp == 0) {
      const double f = calib_first_solve(md, &cal_part[0][0], EPI_WARPS, cal_L, cal_D, cal_c, lane);
      if (lane == 0) cal_fix = f;
    }
    __syncthreads();
    if (own) calib_block<0, 2, EPI_THREADS>(md, mu_s, cal_c, tid, lane, warp, &cal_part[0][0]);
    __syncthreads();
    if (warp == 0) {
      const double f = calib_refine(md, &cal_part[0][0], EPI_WARPS, cal_L, cal_D, cal_c, lane);
      if (lane == 0) cal_fix += f;
    }
    __syncthreads();
    float cpf = 0.f;
    for (int i = own ? tid : md.n_pix; i < md.n_pix; i += EPI_THREADS) {
      const float ms = mu_s[i];
      if (ms == 0.f) continue;
      cpf += calib_pixel_term(md.spec_dn[i] - ms, ms, calib_poly(cal_c, md.calib_n, md.pix_cx[i]));
    }
    double cp = (double)cpf;
#pragma unroll
    for (int o = 16; o; o >>= 1) cp += __shfl_xor_sync(0xffffffffu, cp, o);
    if (lane == 0 && own) red[warp] += cp;
    __syncthreads();
  }
  // photometric terms in FP64, one band per lane of warp 0 (GB300's FP64 pipe
  // is narrow: one warp instruction serves all bands)
  if (warp == 0) {
    double pv = 0.0;
    for (int b = lane; b < md.n_filt; b += 32) {
      const double3 bd = band(b);
      const double is = bd.y;
      if (is != 0.0) {
        const double mn = (double)mb_s[b] * is, dn = bd.x * is;
        const double rr = phot_resid(md, b, dn, mn);
        if (md.floor_bits[0]) {   // sigma_eff of Eq. app_noise_floor
          const double q = floor_q(rs.fl[0], mn, dn, (double)rs.fl[0][3] * is);
          pv += -0.5 * (rr * rr / q + log(q)) + bd.z;
        } else {
          pv += -0.5 * rr * rr + bd.z;
        }
      }
    }
    // the line catalogue (Sec. 3.3), one entry per lane in FP64
    if (LINES)
      for (int k = lane; k < md.n_lcat; k += 32) pv += lcat_term(md, k, ln_F);
#pragma unroll
    for (int o = 16; o; o >>= 1) pv += __shfl_xor_sync(0xffffffffu, pv, o);
    if (lane == 0) {
      double tot = pv;
      for (int w = 0; w < EPI_WARPS && md.n_pix > 0; ++w) tot += red[w];
      if (md.calib_n) tot += cal_fix;
      uint32_t st = 0;
      if (!isfinite(tot)) { st = SED_ROW_NONFINITE; tot = -INFINITY; }
      if (a.lnl) a.lnl[ro] = tot;
      if (a.status) a.status[ro] = st;
    }
  }
}

template <int NT>
cudaError_t launch_epilogue_nt(EpiArgs a, cudaStream_t s) {
  size_t smem = epilogue_smem(a, NT, true);
  a.band_off = (int)epilogue_band_off(a, NT);
  static DynSmemCache set_for[6];
  const bool lines = a.row_model ? a.g.n_line > 0 : a.md.use_lines != 0;
  // age-binned dust and the nebular age axis: neither served nor with lines
  const bool bins = !a.row_model && a.md.n_bin > 0, axis = !a.row_model && a.qneb;
  const int m = bins ? 4 : axis ? 5 : (a.row_model ? 1 : 0) + (lines ? 2 : 0);
  auto k = m == 0 ? k_epilogue<false, false, 0, NT>
         : m == 1 ? k_epilogue<true, false, 0, NT>
         : m == 2 ? k_epilogue<false, true, 0, NT>
         : m == 3 ? k_epilogue<true, true, 0, NT>
         : m == 4 ? k_epilogue<false, false, 1, NT> : k_epilogue<false, false, 2, NT>;
  cudaError_t e = ensure_dyn_smem(k, smem, &set_for[m]);
  if (e == cudaErrorInvalidConfiguration) {   // no room for the bands: they are read where the model keeps them
    a.band_off = 0;
    smem = epilogue_smem(a, NT, false);
    e = ensure_dyn_smem(k, smem, &set_for[m]);
  }
  if (e != cudaSuccess) return e;
  return launch_pdl(k, dim3(a.n), dim3(NT), smem, s, a);
}

cudaError_t launch_epilogue(const EpiArgs& a_in, cudaStream_t s) {
  EpiArgs a = a_in;
  a.lines_off = (int)epilogue_lines_off(a);
  a.samp_off = (int)epilogue_samp_off(a);
  // Threads per row: as many as keep every row of the launch resident at once
  // (1024 threads per SM at 64 registers), where their shared memory fits.
  const int sm = device_sm_count();
  const size_t room = (size_t)220 * 1024;
  if (a.n <= 2 * sm && 2 * epilogue_smem(a, 512, true) <= room) return launch_epilogue_nt<512>(a, s);
  if (a.n <= 4 * sm && 4 * epilogue_smem(a, 256, true) <= room) return launch_epilogue_nt<256>(a, s);
  return launch_epilogue_nt<EPI_THREADS>(a, s);
}

}  // namespace sed
