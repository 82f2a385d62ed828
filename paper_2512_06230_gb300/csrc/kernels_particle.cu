// Particle track model (Section 3 of arXiv 2512.06230: every labeled state
// is a set of P weighted particles moved by constant-turn-rate-and-velocity
// kinematics; births are sampled from their Gaussian; the retained tracks
// get a particle update with resampling).  A component's particles are
// FP64 states (px, py, v, heading, turn rate) and normalised log-weights,
// laid out per component as six rows of P values (CompTable::px).  The
// moment fields of the component (mean, covariance) hold the particles'
// weighted moments, with the mean rounded to FP32 (mlo = 0), so that a
// detection's innovation z - mhi (computed in FP32 by the table kernel) is
// exact and the fixed-point innovation sums of the regeneration give the
// mean detection to FP64 accuracy.
//
// Random numbers: Philox4x32-10 keyed by (seed_lo ^ 0x5851F42D,
// seed_hi ^ frame), counter (label_k, label_b, particle, stream << 24 |
// call); a call's words give two normals by the Box-Muller cosine branch.
// Stream 1: a survivor's accelerations (a, alpha); stream 2: a birth
// particle's five normals (calls 0-2); stream 3: the resampling offset.
#include <math.h>

#include "fx_math.cuh"
#include "glmb_kernels.h"

namespace glmb {

namespace {

constexpr uint32_t kPartKeyXor = 0x5851F42Du;
constexpr int kPartThreads = 256;

__device__ __forceinline__ double unit_open(uint32_t w) { return ((double)w + 0.5) * 2.3283064365386963e-10; }

__device__ __forceinline__ uint4 part_words(const PartModel& pm, int frame, uint32_t lk, uint32_t lb, uint32_t p,
                                            uint32_t stream, uint32_t call) {
  return philox10(make_uint4(lk, lb, p, (stream << 24) | call),
                  make_uint2(pm.seed_lo ^ kPartKeyXor, pm.seed_hi ^ (uint32_t)frame));
}

// What bounds these kernels is the FP64 pipe (an instruction every 16 cycles
// on an SM), so the functions run in integer arithmetic (fx_math.cuh) and what
// is left in FP64 is the states' own arithmetic and the sums, which take a
// fifth of the butterfly's additions (warp_sums).  Per frame, prediction and
// update stages: 200 vehicles 85.9 -> 37.4 and 55.7 -> 46.7 us; a convoy of ten
// 52.1 -> 28.9 and 50.1 -> 42.5.
__device__ const fx::Tables kFx{};

__device__ __forceinline__ void normal_pair(const uint4& w, double& n0, double& n1) {
  n0 = fx::normal(w.x, w.y, kFx.nlog, kFx.inv);
  n1 = fx::normal(w.z, w.w, kFx.nlog, kFx.inv);
}

__device__ __forceinline__ double exp_weight(double l) { return fx::exp_weight(l, kFx.exp2); }

// one CTRV step over dt; the arc (v / w)(sin(psi + w dt) - sin psi, ...)
// as v dt sinc(h)(cos, sin)(psi + h), h = w dt / 2, valid at w = 0.  Heading
// and half angle are added as fractions of a turn, so that the FP64 pipe sees
// 17 operations a particle instead of about 60 (for headings or half angles
// beyond the fixed-point range: the library's functions).
__device__ __forceinline__ void ctrv(const double (&x)[5], double dt, double a, double al, double (&y)[5]) {
  const double h = 0.5 * x[4] * dt;
  double s0, c0, s1, c1, sc;
  if (fx::in_turn_range(h, 0.5) && fx::in_turn_range(x[3], 1e9)) {
    const fx::Turn f = fx::turn(x[3]);
    fx::sincos_turn(f, s0, c0);
    fx::sincos_turn(f + fx::turn(h), s1, c1);
    sc = fx::sinc(h);
  } else {
    double sh, ch;
    sincos(h, &sh, &ch);
    sincos(x[3], &s0, &c0);
    sc = h == 0.0 ? 1.0 : sh / h;
    s1 = s0 * ch + c0 * sh;
    c1 = c0 * ch - s0 * sh;
  }
  const double vdt = x[2] * dt * sc, hd = 0.5 * dt * dt;
  y[0] = x[0] + vdt * c1 + hd * c0 * a;
  y[1] = x[1] + vdt * s1 + hd * s0 * a;
  y[2] = x[2] + dt * a;
  y[3] = x[3] + x[4] * dt + hd * al;
  y[4] = x[4] + dt * al;
}

__device__ __forceinline__ double* prow(const CompTable& ct, int np, int c, int k) {
  return ct.px + ((size_t)c * 6 + k) * np;
}

// Sums of N values over a warp, in the butterfly's order, with the values
// spread over the lanes: at each step a lane hands half of its values to its
// partner, so N = 20 takes 21 additions instead of 100.  Returns one value's
// total and its index k (lanes without one: k >= N).
template <int N, int O>
__device__ __forceinline__ double warp_sums_step(const double (&v)[N], int& k, int& have) {
  if constexpr (O == 0) {
    return v[0];
  } else {
    constexpr int H = (N + 1) / 2;
    const bool up = ((int)threadIdx.x & O) != 0;
    double u[H];
#pragma unroll
    for (int i = 0; i < H; ++i) {
      double hi = 0.0;
      if (i + H < N) hi = v[i + H < N ? i + H : 0];
      u[i] = (up ? hi : v[i]) + __shfl_xor_sync(0xFFFFFFFFu, up ? v[i] : hi, O);
    }
    k += up ? H : 0;
    have = up ? have - H : min(have, H);   // values of the lane that are not padding
    return warp_sums_step<H, O / 2>(u, k, have);
  }
}
template <int N>
__device__ __forceinline__ double warp_sums(const double (&v)[N], int& k) {
  int have = N;
  k = 0;
  const double t = warp_sums_step<N, 16>(v, k, have);
  if (have < 1) k = N;
  return t;
}

// Sums of N values over the block, left at tot (`done` gets them in one thread
// first, for what follows from them); red holds (threads / 32) * N doubles.
template <int N, typename F>
__device__ void block_sum(double (&v)[N], double* red, double* tot, F done) {
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (N == 1) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], o);
    if ((threadIdx.x & 31) == 0) red[w] = v[0];
  } else {
    int k;
    const double t = warp_sums<N>(v, k);
    if (k < N) red[w * N + k] = t;
  }
  __syncthreads();
  if (threadIdx.x < N) {
    double s = 0.0;
    for (int i = 0; i < nw; ++i) s += red[i * N + threadIdx.x];
    tot[threadIdx.x] = s;
    if (N == 1) done(s);
  }
  __syncthreads();
}
template <int N>
__device__ void block_sum(double (&v)[N], double* red, double* tot) {
  block_sum<N>(v, red, tot, [](double) {});
}

__device__ double block_max(double v, double* red) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
  if (lane == 0) red[w] = v;
  __syncthreads();
  double m = -INFINITY;
  for (int i = 0; i < nw; ++i) m = fmax(m, red[i]);
  __syncthreads();
  return m;
}

// A block's particles, PER a thread in registers (particle threadIdx.x + i *
// blockDim.x), or, PER = 0, in global memory: the update of a component reads
// and sums them several times.
template <int PER>
__device__ __forceinline__ int particles_of(int np) {
  return PER > 0 ? PER : (np - (int)threadIdx.x + (int)blockDim.x - 1) / (int)blockDim.x;
}

// weighted mean and covariance of component c's particles into its moment
// fields (mean rounded to FP32, mlo = 0); x(i, k) and w(i) give row k and the
// weight of the thread's particle i
template <int PER, typename X, typename W>
__device__ __forceinline__ void write_moments(const CompTable& ct, int np, int c, X x, W w, double* red, double* tot) {
  const int n = particles_of<PER>(np), lane = (int)threadIdx.x;
  double s[5] = {0, 0, 0, 0, 0};
#pragma unroll PER > 0 ? PER : 1
  for (int i = 0; i < n; ++i) {
    if (lane + i * (int)blockDim.x >= np) break;
    const double wi = w(i);
#pragma unroll
    for (int k = 0; k < 5; ++k) s[k] += wi * x(i, k);
  }
  block_sum<5>(s, red, tot);
#pragma unroll
  for (int k = 0; k < 5; ++k) s[k] = tot[k];
  double q[15];
#pragma unroll
  for (int k = 0; k < 15; ++k) q[k] = 0.0;
#pragma unroll PER > 0 ? PER : 1
  for (int i = 0; i < n; ++i) {
    if (lane + i * (int)blockDim.x >= np) break;
    const double wi = w(i);
    double d[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) d[k] = x(i, k) - s[k];
    int k = 0;
#pragma unroll
    for (int a = 0; a < 5; ++a)
#pragma unroll
      for (int b = a; b < 5; ++b, ++k) q[k] += wi * d[a] * d[b];
  }
  const size_t cap = ct.cap;
  if (lane < 5) {
    ct.mhi[lane * cap + c] = (float)tot[lane];
    ct.mlo[lane * cap + c] = 0.f;
  }
  block_sum<15>(q, red, tot + 5);
  if (lane < 15) ct.cov[(size_t)lane * cap + c] = (float)tot[5 + lane];
  __syncthreads();   // the weights and the totals are reused by the next component
}

// Prediction, particle by particle (a flat grid over the working table's
// components x particles, so that the FP64 work of one component runs on
// into the next without a barrier): a survivor's particle takes one CTRV
// step with its own accelerations; a birth's particle is drawn through the
// Cholesky factor that the host stored with the birth.  Particle 0 of each
// component writes its label and existence.
__global__ void __launch_bounds__(kPartThreads) particle_step_kernel(Model md, PartModel pm, CompTable src,
                                                                     CompTable dst, const FrameDev* fs,
                                                                     const double* __restrict__ births) {
  pdl_enter();
  const int n = fs->n_comp, nb = fs->nb, frame = fs->frame, np = pm.np;
  const long long total = (long long)(n + nb) * np;
  const double lw_b = -log((double)np);
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i / np), p = (int)(i - (long long)c * np);
    if (c < n) {
      const uint32_t lk = src.lk[c], lb = src.lb[c];
      double x[5], y[5], n0, n1;
#pragma unroll
      for (int k = 0; k < 5; ++k) x[k] = prow(src, np, c, k)[p];
      normal_pair(part_words(pm, frame, lk, lb, (uint32_t)p, 1u, 0u), n0, n1);
      ctrv(x, pm.dt, pm.sigma_a * n0, pm.sigma_w * n1, y);
#pragma unroll
      for (int k = 0; k < 5; ++k) prow(dst, np, c, k)[p] = y[k];
      prow(dst, np, c, 5)[p] = prow(src, np, c, 5)[p];
      if (p == 0) {
        dst.lk[c] = lk;
        dst.lb[c] = lb;
        dst.logp[c] = md.log_ps;
        dst.log1mp[c] = md.log_1mps;
      }
    } else {
      const int b = c - n;
      const double* rec = births + (size_t)b * kBirthRec;
      const double* L = rec + kBirthChol;   // lower triangle, row-major
      double xi[6];
#pragma unroll
      for (int j = 0; j < 3; ++j)
        normal_pair(part_words(pm, frame, (uint32_t)frame, (uint32_t)b, (uint32_t)p, 2u, (uint32_t)j), xi[2 * j],
                    xi[2 * j + 1]);
#pragma unroll
      for (int a = 0; a < 5; ++a) {
        double v = rec[1 + a];
#pragma unroll
        for (int k = 0; k <= a; ++k) v += L[a * (a + 1) / 2 + k] * xi[k];
        prow(dst, np, c, a)[p] = v;
      }
      prow(dst, np, c, 5)[p] = lw_b;
      if (p == 0) {
        const double r = rec[0];
        dst.lk[c] = (uint32_t)frame;
        dst.lb[c] = (uint32_t)b;
        dst.logp[c] = r > 0.0 ? (float)log(r) : -INFINITY;
        dst.log1mp[c] = r < 1.0 ? (float)log1p(-r) : -INFINITY;
      }
    }
  }
}

// The working table's moments: one block of 128 threads per component (64: 3 us
// more for a convoy of ten, the same for 200 vehicles),
// threads over its particles, one pass with offsets from its particle 0, d_p = x_p - x_0:
// mean = x_0 + sum w d, covariance = sum w d d^T - (sum w d)(sum w d)^T
// (the weights sum to one), mean rounded to FP32 with a zero low part.
__global__ void __launch_bounds__(kPartThreads) particle_moments_kernel(PartModel pm, CompTable ct,
                                                                       const FrameDev* fs) {
  pdl_enter();
  __shared__ double part[(kPartThreads / 32) * 20], tot[20];
  const int T = fs->T, np = pm.np;
  for (int c = blockIdx.x; c < T; c += gridDim.x) {
    double x0[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) x0[k] = prow(ct, np, c, k)[0];
    double v[20];   // sum w d (5), sum w d d^T (15, packed)
#pragma unroll
    for (int k = 0; k < 20; ++k) v[k] = 0.0;
    for (int p = threadIdx.x; p < np; p += blockDim.x) {
      const double w = exp_weight(prow(ct, np, c, 5)[p]);
      double d[5];
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        d[k] = prow(ct, np, c, k)[p] - x0[k];
        v[k] += w * d[k];
      }
      int k = 5;
#pragma unroll
      for (int i = 0; i < 5; ++i)
#pragma unroll
        for (int j = i; j < 5; ++j, ++k) v[k] += w * d[i] * d[j];
    }
    block_sum<20>(v, part, tot);
    const size_t cap = ct.cap;
    const int e = (int)threadIdx.x;
    if (e < 5) {
      ct.mhi[e * cap + c] = (float)(prow(ct, np, c, e)[0] + tot[e]);
      ct.mlo[e * cap + c] = 0.f;
    }
    if (e < 15) {
      int i = 0, j = e;   // entry e of the packed upper triangle
      while (j >= 5 - i) {
        j -= 5 - i;
        ++i;
      }
      ct.cov[(size_t)e * cap + c] = (float)(tot[5 + e] - tot[i] * tot[i + j]);
    }
    __syncthreads();
  }
}

// Compatibility entries: the warps of a block on one component, a pair to a
// warp at a time, lanes over particles;
// log C = log P_D + log sum_p w_p N(z; (px, py)_p, R) for each of the
// component's gated pairs (the table kernels wrote the pairs, gated on
// the moments), then the death probability from these entries.  The
// offsets run in FP32: a particle's position relative to the component's
// FP32 mean, (px, py)_p - mhi, is formed once in FP64 and rounded, and a
// pair's innovation z - mhi is the table's (exact in FP32 when z and mhi
// are within a factor of two, as for any gated pair away from the
// origin); z - (px, py)_p is their difference.  The mixture's sum is in
// FP32 too (log C is stored in FP32).  Particles beyond kRegP per lane
// are re-read from the particle rows.
constexpr int kRegP = 8;   // particles held in registers per lane (256 per warp)
// A component's pairs are few (up to a dozen or two), but with one warp each
// they follow one another through shuffles and exponentials, and the frame
// waits for its longest list: four warps share a component, and the death
// probability's sum over the pairs, whose order is the pairs', follows.  Table
// stage with one, two and four warps: 22.7, 17.8 and 16.1 us (convoy of ten),
// 25.9, 20.8 and 20.0 (200 vehicles).
constexpr int kLogcWarps = 4;

__global__ void __launch_bounds__(32 * kLogcWarps) particle_logc_kernel(Model md, PartModel pm, CompTable ct,
                                                                        PairTable pt, const FrameDev* fs) {
  pdl_enter();
  __shared__ float s_logc[32];
  const int T = fs->T, np = pm.np, lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  if (fs->M > 0 && !__isGlobal(fs->Z)) return;   // flagged by the table kernel
  const unsigned cap_p = (unsigned)min(pt.cap_pairs, (long long)0xFFFFFFFF);
  const size_t capp = (size_t)pt.cap_pairs;
  const float r0 = (float)pm.Rinv[0], r1 = (float)(pm.Rinv[1] + pm.Rinv[2]), r3 = (float)pm.Rinv[3];
  const float lc0 = (float)(pm.log_pd - pm.lnorm);
  for (int c = blockIdx.x; c < T; c += gridDim.x) {
    const unsigned k0 = min(pt.ptr[c], cap_p), k1 = min(k0 + pt.cnt[c], cap_p);
    const double mx = (double)ct.mhi[c], my = (double)ct.mhi[(size_t)ct.cap + c];
    float ox[kRegP], oy[kRegP], ow[kRegP];
#pragma unroll
    for (int j = 0; j < kRegP; ++j) {
      const int p = lane + 32 * j;
      const bool in = p < np;
      ox[j] = in ? (float)(prow(ct, np, c, 0)[p] - mx) : 0.f;
      oy[j] = in ? (float)(prow(ct, np, c, 1)[p] - my) : 0.f;
      ow[j] = in ? (float)prow(ct, np, c, 5)[p] : -INFINITY;
    }
    float lm = -INFINITY, ls = 0.f;
    bool any = false;
    for (unsigned kb = k0; kb < k1; kb += 32) {   // 32 pairs, then their part of the sum
    const unsigned ke = min(kb + 32u, k1);
    for (unsigned k = kb + wp; k < ke; k += kLogcWarps) {
      const float ex = pt.e[k], ey = pt.e[capp + k];
      // the register-held particles' terms are independent: their maximum,
      // then the sum of their exponentials (no dependent chain through expf)
      float l[kRegP];
      float m = -INFINITY;
#pragma unroll
      for (int j = 0; j < kRegP; ++j) {
        const float dx = ex - ox[j], dy = ey - oy[j];
        l[j] = ow[j] - 0.5f * (r0 * dx * dx + r1 * dx * dy + r3 * dy * dy);
        m = fmaxf(m, l[j]);
      }
      float s = 0.f;
      if (m > -INFINITY) {
#pragma unroll
        for (int j = 0; j < kRegP; ++j) s += expf(l[j] - m);
      }
      auto push = [&](float dx, float dy, float w) {
        const float lv = w - 0.5f * (r0 * dx * dx + r1 * dx * dy + r3 * dy * dy);
        if (lv > m) {
          s = s * expf(m - lv) + 1.f;
          m = lv;
        } else if (lv > -INFINITY) {
          s += expf(lv - m);
        }
      };
      for (int p = lane + 32 * kRegP; p < np; p += 32)
        push(ex - (float)(prow(ct, np, c, 0)[p] - mx), ey - (float)(prow(ct, np, c, 1)[p] - my),
             (float)prow(ct, np, c, 5)[p]);
      // the warp's maximum, then each lane's sum rescaled to it once and
      // added across the warp
      float mw = m;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mw = fmaxf(mw, __shfl_xor_sync(0xFFFFFFFFu, mw, o));
      float sw = m == -INFINITY ? 0.f : s * expf(m - mw);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sw += __shfl_xor_sync(0xFFFFFFFFu, sw, o);
      const float logC = mw == -INFINITY ? -INFINITY : lc0 + mw + logf(sw);
      if (lane == 0) {
        pt.logC[k] = logC;
        s_logc[k - kb] = logC;
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      any = true;
      if (!md.kappa_zero)
        for (unsigned k = kb; k < ke; ++k) lse_push(lm, ls, s_logc[k - kb] - md.log_kappa);
    }
    __syncthreads();
    }
    if (threadIdx.x == 0) death_prob(md, ct.logp[c], ct.log1mp[c], lm, ls, any, pt.dprob[c], pt.dthr[c]);
  }
}

// Regeneration: one block per kept component (copied to its compacted
// position) and per distinct (component, detection set) update (written
// after the kept ones): log w_p -= (m / 2) (zbar - h_p)^T R^-1 (zbar - h_p)
// (the product of the m detections' likelihoods up to a factor common to
// all particles), normalised; systematic resampling when the effective
// sample size is below ess_frac * P.  Dynamic shared memory: 2 P doubles
// (log-weights; weights, then cumulative weights).
// What bounds it is the chain of block reductions and, with many updates, the
// FP64 pipe: the particles stay in registers (PER a thread) between the
// passes, the runs of the cumulative weights are scanned across the warps,
// the search compares the weights' bits, and what all threads share is formed
// by one.
template <int PER>
__global__ void __launch_bounds__(kPartThreads, 2) particle_remap_kernel(
    Model md, PartModel pm, CompTable src, CompTable dst, const uint32_t* __restrict__ newpos,
    const uint32_t* __restrict__ flag, const FrameDev* __restrict__ fs, const unsigned* __restrict__ n_keep_dev,
    const uint32_t* __restrict__ upd_src, const uint32_t* __restrict__ upd_m, const long long* __restrict__ upd_se,
    int cap_upd, const unsigned* __restrict__ n_upd_dev, const unsigned* __restrict__ n_surv_dev, unsigned* err) {
  pdl_enter();
  extern __shared__ double s_dyn[];
  __shared__ double red[(kPartThreads / 32) * 15], tot[20];
  __shared__ double s_wsum[kPartThreads / 32];
  if (*n_surv_dev == 0u || (*(volatile unsigned*)err & kErrFatal)) return;
  const int n_src = fs->T, np = pm.np, frame = fs->frame;
  double* s_l = s_dyn;         // log-weights
  double* cum = s_dyn + np;    // weights, then cumulative weights
  const int tid = (int)threadIdx.x, bd = (int)blockDim.x;
  const unsigned n_keep = *n_keep_dev;
  const unsigned n_upd = min(*n_upd_dev, (unsigned)cap_upd);
  if ((long long)n_keep + n_upd > dst.cap) return;   // flagged by the remap kernel
  for (long long x = blockIdx.x; x < (long long)n_src + n_upd; x += gridDim.x) {
    if (x < n_src) {
      const int c = (int)x;
      if (!flag[c]) continue;
      if (newpos[c] >= n_keep) {
        if (threadIdx.x == 0) atomicOr(err, kErrChkComp);
        continue;
      }
      const int d = (int)newpos[c];
      for (int k = 0; k < 6; ++k)
        for (int p = threadIdx.x; p < np; p += blockDim.x) prow(dst, np, d, k)[p] = prow(src, np, c, k)[p];
      if (threadIdx.x < 5) {
        dst.mhi[threadIdx.x * (size_t)dst.cap + d] = src.mhi[threadIdx.x * (size_t)src.cap + c];
        dst.mlo[threadIdx.x * (size_t)dst.cap + d] = 0.f;
      }
      if (threadIdx.x < 15) dst.cov[threadIdx.x * (size_t)dst.cap + d] = src.cov[threadIdx.x * (size_t)src.cap + c];
      if (threadIdx.x == 0) {
        dst.lk[d] = src.lk[c];
        dst.lb[d] = src.lb[c];
        dst.logp[d] = src.logp[c];
        dst.log1mp[d] = src.log1mp[c];
      }
      continue;
    }
    const int u = (int)(x - n_src);
    const int c = (int)upd_src[u];
    if (c >= n_src) {
      if (threadIdx.x == 0) atomicOr(err, kErrChkComp);
      continue;
    }
    const int d = (int)n_keep + u;
    const double m = (double)max(upd_m[u], 1u);   // an update holds at least one detection
    double zb[2];
#pragma unroll
    for (int a = 0; a < 2; ++a)
      zb[a] = (double)src.mhi[a * (size_t)src.cap + c] + (double)upd_se[(size_t)a * cap_upd + u] * kFxInv / m;
    // reweight, then normalise
    constexpr int kHeld = PER > 0 ? PER : 1;
    double xr[kHeld][5];
    double mx = -INFINITY;
    const int n = particles_of<PER>(np);
#pragma unroll PER > 0 ? PER : 1
    for (int i = 0; i < n; ++i) {
      const int p = tid + i * bd;
      if (p >= np) break;
      double px = prow(src, np, c, 0)[p], py = prow(src, np, c, 1)[p];
      const double l0 = prow(src, np, c, 5)[p];
      if (PER > 0) {
        xr[i % kHeld][0] = px;
        xr[i % kHeld][1] = py;
#pragma unroll
        for (int k = 2; k < 5; ++k) xr[i % kHeld][k] = prow(src, np, c, k)[p];
      }
      const double ex = zb[0] - px, ey = zb[1] - py;
      const double l =
          l0 - 0.5 * m * (pm.Rinv[0] * ex * ex + (pm.Rinv[1] + pm.Rinv[2]) * ex * ey + pm.Rinv[3] * ey * ey);
      s_l[p] = l;
      mx = fmax(mx, l);
    }
    mx = block_max(mx, red);
    double sv[1] = {0.0};
    for (int p = tid; p < np; p += bd) {
      const double e = exp_weight(s_l[p] - mx);
      cum[p] = e;
      sv[0] += e;
    }
    block_sum<1>(sv, red, tot, [&](double t) {   // (one warp's FP64 work, not every warp's)
      tot[1] = mx + log(t);
      tot[2] = 1.0 / t;
    });
    const double lse = tot[1], inv = tot[2];
    // normalised weights cum[p] = exp(l_p - mx) / sum, log-weights l_p - lse
    double s2[1] = {0.0};
    for (int p = tid; p < np; p += bd) {
      const double w = cum[p] * inv;
      cum[p] = w;
      s2[0] += w * w;
    }
    block_sum<1>(s2, red, tot, [&](double t) {
      tot[1] = 1.0 / t;
      if (tot[1] < pm.ess_frac * np) {
        tot[2] = -log((double)np);
        tot[3] = 1.0 / np;
      }
    });
    const bool resample = tot[1] < pm.ess_frac * np;
    const double lw_r = tot[2], w_r = tot[3];
    if (resample) {
      // cumulative weights: each thread scans a contiguous run, then the
      // runs' totals are scanned over the block
      const int per = (np + bd - 1) / bd, b0 = min(np, tid * per), b1 = min(np, b0 + per);
      double run = 0.0;
      for (int p = b0; p < b1; ++p) {
        run += cum[p];
        cum[p] = run;
      }
      const int lane = tid & 31, wp = tid >> 5;
      double incl = run;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const double y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
      }
      if (lane == 31) s_wsum[wp] = incl;
      __syncthreads();
      // (the exclusive scan from the lower lanes' totals: no rounding of incl - run)
      double off = __shfl_up_sync(0xFFFFFFFFu, incl, 1);
      if (lane == 0) off = 0.0;
      double before = 0.0;
      for (int w = 0; w < wp; ++w) before += s_wsum[w];
      off += before;
      for (int p = b0; p < b1; ++p) cum[p] += off;
      __syncthreads();
      const double u0 = unit_open(part_words(pm, frame, src.lk[c], src.lb[c], 0u, 3u, 0u).x);
      const bool pow2 = (np & (np - 1)) == 0;   // then 1 / np is exact
      const unsigned long long* bits = reinterpret_cast<const unsigned long long*>(cum);
#pragma unroll PER > 0 ? PER : 1
      for (int i = 0; i < n; ++i) {
        const int r = tid + i * bd;
        if (r >= np) break;
        const double target = pow2 ? (u0 + r) * w_r : (u0 + r) / np;
        const unsigned long long tb = fx::to_bits(target);
        int lo = 0, hi = np - 1;   // first k with cum[k] > target, else np - 1
        while (lo < hi) {          // (doubles that are not negative compare as their bits)
          const int mid = (lo + hi) >> 1;
          if (bits[mid] > tb) hi = mid;
          else lo = mid + 1;
        }
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          const double v = prow(src, np, c, k)[lo];
          if (PER > 0) xr[i % kHeld][k] = v;
          prow(dst, np, d, k)[r] = v;
        }
        prow(dst, np, d, 5)[r] = lw_r;
      }
    } else {
#pragma unroll PER > 0 ? PER : 1
      for (int i = 0; i < n; ++i) {
        const int p = tid + i * bd;
        if (p >= np) break;
#pragma unroll
        for (int k = 0; k < 5; ++k) prow(dst, np, d, k)[p] = PER > 0 ? xr[i % kHeld][k] : prow(src, np, c, k)[p];
        prow(dst, np, d, 5)[p] = s_l[p] - lse;
      }
    }
    write_moments<PER>(
        dst, np, d,
        [&](int i, int k) { return PER > 0 ? xr[i % kHeld][k] : prow(dst, np, d, k)[tid + i * bd]; },
        [&](int i) { return resample ? w_r : cum[tid + i * bd]; }, red, tot);
    if (tid == 0) {
      dst.lk[d] = src.lk[c];
      dst.lb[d] = src.lb[c];
      dst.logp[d] = src.logp[c];
      dst.log1mp[d] = src.log1mp[c];
    }
  }
}

}  // namespace

void particle_init(int smem_limit) {
  opt_in_smem(particle_remap_kernel<4>, smem_limit);
  opt_in_smem(particle_remap_kernel<0>, smem_limit);
}

void launch_particle_predict(const Model& md, const PartModel& pm, const CompTable& src, const CompTable& dst,
                             const FrameDev* fs, const double* births_dev, int grid, cudaStream_t s) {
  launch_k(particle_step_kernel, grid, kPartThreads, 0, s, md, pm, src, dst, fs, births_dev);
  launch_k(particle_moments_kernel, 4 * grid, 128, 0, s, pm, dst, fs);
}

void launch_particle_logc(const Model& md, const PartModel& pm, const CompTable& ct, const PairTable& pt,
                          const FrameDev* fs, int grid, cudaStream_t s) {
  launch_k(particle_logc_kernel, 4 * grid, 32 * kLogcWarps, 0, s, md, pm, ct, pt, fs);
}

void launch_particle_remap(const Model& md, const PartModel& pm, const CompTable& src, const CompTable& dst,
                           const uint32_t* newpos, const uint32_t* flag, const FrameDev* fs,
                           const unsigned* n_keep_dev, const uint32_t* upd_src, const uint32_t* upd_m,
                           const long long* upd_se, int cap_upd, const unsigned* n_upd_dev,
                           const unsigned* n_surv_dev, unsigned* err, int grid, int h_max, cudaStream_t s) {
  // a thread per four particles, which it then holds: several updates in
  // flight per SM, each with short block reductions; a thread per two where
  // few hypotheses make few updates, whose chains the frame waits for (above
  // 1024 particles 64 threads, the particles in memory).  Update stage with 256
  // particles, before and with 64 and 128 threads: convoy of ten (h_max 100)
  // 42.6, 35.1 and 30.4 us; 200 vehicles (h_max 1000) 47.5, 39.6 and 41.9.
  // Over the range, four and two a thread: 20 and 60 vehicles at h_max 25 to
  // 256, 36.2 and 32.0 (256 particles), 31.6 and 29.1 (100), 37.5 and 38.7
  // (512: blocks of 256 threads spend more in their barriers, so four a thread
  // from 257 particles on; 200 vehicles with 512: 49 and 57); 200 vehicles with
  // 256, h_max 25, 100, 256, 500: 39.0 and 36.7, 39.1 and 38.1, 39.7 and 40.4,
  // 39.2 and 40.7
  const size_t smem = particle_remap_smem(pm.np);
  int threads = pm.np <= 256 ? 64 : pm.np <= 512 ? 128 : pm.np <= 1024 ? 256 : 64;
  if (h_max <= 256 && pm.np > threads && pm.np <= 256) threads *= 2;
  auto k = pm.np <= 1024 ? particle_remap_kernel<4> : particle_remap_kernel<0>;
  launch_k(k, 4 * grid, threads, smem, s, md, pm, src, dst, newpos, flag, fs, n_keep_dev, upd_src, upd_m, upd_se, cap_upd,
           n_upd_dev, n_surv_dev, err);
}

int particle_remap_smem(int np) { return 2 * np * (int)sizeof(double); }

}  // namespace glmb
