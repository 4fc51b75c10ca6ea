// Real-space electrode-ion sums of the potential, the slab dipole term, and
// b = chi - k_e b^sol (Eq. 25): sum over the images within r_c of
// q_I [erfc(g r) - erfc(alpha_i r)] / r.
//
// A warp holds 32 electrode atoms (one a lane) and goes over a share of the frame's ions on
// its own.  It reads 32 ions at a time, drops those that no image of its atoms' bounding box
// can reach (a lane an ion), and screens the rest for every lane at once in float.  Each
// lane keeps the pairs that pass in a list of its own in shared memory, and the warp
// evaluates the lists' heads together, each lane adding to its own atom's sum: no
// compaction, no exchange of values between lanes.
//
// Float storage evaluates near pairs in float pairs (hi + lo, ~1e-12 of the pair: the
// difference from 64-bit fixed-point coordinates, erfc(x)/x from a table) and far ones, where
// erfc(g r) / r <= 1e-4 1/A, in plain float from the fixed-point difference (~1e-6 of a term,
// <= 1e-10 1/A; three quarters of the images at a third of the instructions).  FP64 runs at
// 1/64 of the float rate here and an FP64 erfc is some fifty operations, which is what
// bound the kernel before: with near pairs in FP64, both kinds through queues of the warp,
// every ion screened by every lane, it took 16.4 ms at 26,600 atoms, 5,000 ions and 16 frames
// (r_c 24 A, 550 images an atom) against 1.81 ms; 183 against 14 us at 12,800 atoms, 2,000
// ions and one frame; 121 against 12 us at 512 atoms and 200 ions, where four blocks held all
// the work; 2.57 against 1.45 ms at 512 atoms, 2,000 ions, 256 frames (three images a pair).
// FP64 storage evaluates every image in FP64.
#include <math.h>

#include <algorithm>
#include <vector>

#include "phasor.cuh"
#include "programmatic.cuh"

namespace cpm {

namespace {

// ---- H(s) = erfc(sqrt s) / sqrt s on [2^-8, 2^6) -----------------------------------------
// erfc(g r) / r = g H(g^2 r^2) for any g, so one table serves the Ewald and the Gaussian
// term of every atom.  64 intervals an octave; in each the degree-5 interpolant at the
// Chebyshev nodes, as a polynomial in s - (interval centre): (c0 hi, c0 lo, c1 hi, c1 lo),
// (c2, c3, c4, c5).  |t| / s <= 1/128, so the float terms c2 t^2 .. carry 6e-5 of the value
// and their rounding 4e-12 of it; the interpolation error is below 1e-12.
constexpr int kHOctaves = 14, kHFirst = -8, kHPer = 64;
constexpr int kHIntervals = kHOctaves * kHPer;
constexpr float kHMin = 0.00390625f;  // 2^-8

std::vector<float> make_h_table() {
  std::vector<float> tab(8 * kHIntervals);
  constexpr int kDeg = 5;
  for (int i = 0; i < kHIntervals; ++i) {
    const double oct = ldexp(1.0, kHFirst + i / kHPer);
    const double half = oct / (2 * kHPer);
    const double x0 = oct + (2 * (i % kHPer) + 1) * half;
    // Newton's divided differences at the nodes (in units of the half width), then expanded
    double u[kDeg + 1], c[kDeg + 1], p[kDeg + 1] = {0};
    for (int k = 0; k <= kDeg; ++k) {
      u[k] = cos(kPi * (2 * k + 1) / (2 * (kDeg + 1)));
      const double r = sqrt(x0 + u[k] * half);
      c[k] = erfc(r) / r;
    }
    for (int k = 1; k <= kDeg; ++k)
      for (int j = kDeg; j >= k; --j) c[j] = (c[j] - c[j - 1]) / (u[j] - u[j - k]);
    for (int k = kDeg; k >= 0; --k) {  // p = p (x - u_k) + c_k
      for (int j = kDeg; j > 0; --j) p[j] = p[j - 1] - u[k] * p[j];
      p[0] = c[k] - u[k] * p[0];
    }
    double scale = 1.0;
    for (int j = 0; j <= kDeg; ++j, scale /= half) p[j] *= scale;
    float* t = &tab[8 * i];
    t[0] = (float)p[0];
    t[1] = (float)(p[0] - (double)t[0]);
    t[2] = (float)p[1];
    t[3] = (float)(p[1] - (double)t[2]);
    for (int j = 2; j <= kDeg; ++j) t[2 + j] = (float)p[j];
  }
  return tab;
}

// (h, l) = H(sh + sl) for kHMin <= sh < 2^6.
__device__ __forceinline__ void h_table(const float4* __restrict__ T, float sh, float sl,
                                        float& h, float& l) {
  const uint32_t bits = __float_as_uint(sh);
  const int i = (int)(bits >> 17) - ((127 + kHFirst) << 6);
  const float x0 = __uint_as_float((bits & 0xFFFE0000u) | 0x00010000u);
  const float4 a = __ldg(T + 2 * i), b = __ldg(T + 2 * i + 1);
  const float t = sh - x0;  // exact
  const float tf = t + sl;
  const float m = __fmul_rn(a.z, t);
  const float me = fmaf(a.z, t, -m);
  const float p = fmaf(tf, fmaf(tf, fmaf(tf, b.w, b.z), b.y), b.x);
  const float lo = fmaf(tf * tf, p, fmaf(a.z, sl, fmaf(a.w, t, a.y)) + me);
  h = a.x + m;
  l = (a.x - h) + m + lo;
}

// ---- records -----------------------------------------------------------------------------
// A point's fractional coordinates in 64-bit fixed point: x, y, z hold them rounded to
// 2^-32, xl, yl, zl the signed rest in 2^-64.  Ions: (qh, ql) = q as a float pair.
struct IonRec {
  uint32_t x, y, z;
  float qh;
  int32_t xl, yl, zl;
  float ql;
};

// Atoms: (ah, al) = alpha^2 and (bh, bl) = -alpha / g as float pairs.
struct AtomRec {
  int32_t xl, yl, zl;
  float ah, al, bh, bl, pad;
};

__device__ __forceinline__ void fixed64(double x, double L, uint32_t& hi, int32_t& lo) {
  double s = x / L;
  s -= floor(s);
  hi = (uint32_t)((unsigned long long)llrint(s * 4294967296.0) & 0xffffffffull);
  const unsigned long long u = (unsigned long long)(s * 18446744073709551616.0);
  const long long r = (long long)(u - ((unsigned long long)hi << 32));
  lo = (int32_t)(r > 2147483647ll ? 2147483647ll : r < -2147483648ll ? -2147483648ll : r);
}

__device__ __forceinline__ void split(double v, float& h, float& l) {
  h = (float)v;
  l = isfinite(h) ? (float)(v - (double)h) : 0.f;
}

constexpr int kPrepThreads = 128;

// The ions' fixed-point coordinates (the phases of every k-vector use them), their records,
// and the block's sums of q z and q for the dipole term and Q^sol: sums[frame][block].  Fixed point
// has no place for a coordinate that is not finite: the frame's sum of q z is NaN then, and so are
// its b.
__global__ void __launch_bounds__(kPrepThreads)
k_ion_prepare(const double* __restrict__ ion_xyz, const double* __restrict__ ion_q, int n_ion,
              double lx, double ly, double lz, uint32_t* __restrict__ sion,
              IonRec* __restrict__ rec, double2* __restrict__ sums, unsigned* far_state,
              unsigned long long* stamp) {
  __shared__ double2 red[kPrepThreads / 32];
  set_up_next();
  stamp_time(stamp);
  if (far_state && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 2)
    far_state[threadIdx.x] = 0u;
  const int f = blockIdx.y, t = blockIdx.x * kPrepThreads + threadIdx.x;
  double qz = 0.0, qs = 0.0;
  if (t < n_ion) {
    const size_t e = (size_t)f * n_ion + t;
    IonRec r;
    const double x = ion_xyz[3 * e], y = ion_xyz[3 * e + 1], z = ion_xyz[3 * e + 2], q = ion_q[e];
    fixed64(x, lx, r.x, r.xl);
    fixed64(y, ly, r.y, r.yl);
    fixed64(z, lz, r.z, r.zl);
    split(q, r.qh, r.ql);
    sion[3 * e] = r.x;
    sion[3 * e + 1] = r.y;
    sion[3 * e + 2] = r.z;
    rec[e] = r;
    qz = isfinite(x) && isfinite(y) && isfinite(z) ? q * z : nan("");
    qs = q;
  }
  for (int o = 16; o; o >>= 1) {
    qz += __shfl_xor_sync(0xffffffffu, qz, o);
    qs += __shfl_xor_sync(0xffffffffu, qs, o);
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = make_double2(qz, qs);
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kPrepThreads / 32; ++w) {
      qz += red[w].x;
      qs += red[w].y;
    }
    sums[(size_t)f * gridDim.x + blockIdx.x] = make_double2(qz, qs);
  }
}

__global__ void k_atom_records(const double* __restrict__ xyz, const double* __restrict__ alpha,
                               int n, double lx, double ly, double lz, double g,
                               AtomRec* __restrict__ rec) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  AtomRec r;
  uint32_t hi;
  fixed64(xyz[3 * i], lx, hi, r.xl);
  fixed64(xyz[3 * i + 1], ly, hi, r.yl);
  fixed64(xyz[3 * i + 2], lz, hi, r.zl);
  split(alpha[i] * alpha[i], r.ah, r.al);
  split(-alpha[i] / g, r.bh, r.bl);
  r.pad = 0.f;
  rec[i] = r;
}

// ---- the sums ----------------------------------------------------------------------------

constexpr int kMaxShifts = 64;
constexpr int kFarTerms = 16;  // far terms of each lane that a block of the pool holds
constexpr int kRealWarps = 8;
constexpr int kListDepth = 72;  // pairs a lane can hold: fewer than 64 at a look, and at
constexpr int kListStep = 8;    // most this many more before the next one
// an entry of a list: shift << kIonBits | ion, the ion relative to a base moved on when full
template <int kMode>
constexpr int kIonBits = 16;

// Screen modes: every box edge above 2 r_c (the nearest image only), a list of whole-box
// shifts of the nearest image (each its own pair), or every image of a screened pair in FP64
// (boxes so small that more than kMaxShifts shifts would be needed).
enum RealMode { kSingleImage = 0, kShiftList = 1, kAllImages = 2 };

template <>
constexpr int kIonBits<kShiftList> = 10;

struct RealArgs {
  const double *xyz, *alpha;   // electrode
  const uint32_t* sfix;
  const AtomRec* atoms;
  int n;
  const double *ion_xyz, *ion_q;
  const IonRec* ions;
  int n_ion, shares;           // shares of the ions: warps of a block that split them
  const float4* htab;
  double L[3], invL[3], g, rc, rc2;
  bool single[3];              // edge above 2 r_c
  float fs[3], fsh[3], fsl[3]; // L / 2^32: float, and as a float pair
  float reach[3];              // L / 2 - r_c: largest half extent of a box of atoms whose
                               // ions need no wrapping (see below)
  float screen2;               // r_c^2 + 0.01
  float far2, cut2;            // far images: r_split^2 <= r^2 < r_c^2 (1 - 1e-5)
  float rc2h, rc2l, g2h, g2l;  // r_c^2, g^2 and g as float pairs
  float gh, gl;
  int nshift;
  float shift[kMaxShifts][3];  // k L, the screen's
  signed char kshift[kMaxShifts][3];
  double* part;                // [gridDim.z][frames][n]
  // far terms of a share in the ions' order (far_blocks 0: summed by the share), in blocks
  // of a pool [far_blocks][kFarTerms][32] that a warp takes as its lists grow:
  float* far;
  unsigned* far_state;  // blocks taken, whether more were wanted than there are
  int* far_row;         // [share][frame][group][far_len]: the warp's blocks
  int* far_count;       // [share][frame][group][32]
  int far_blocks, far_len;
};

// FP64 sum of one electrode-ion pair over every image within r_c.
__device__ __forceinline__ double pair_images(const double* ri, double ai, const double* ion,
                                              double q, const RealArgs& a) {
  double d[3];
  int lo[3], hi[3];
  for (int u = 0; u < 3; ++u) {
    d[u] = ri[u] - ion[u];
    if (a.single[u]) {  // box edge above 2 rc: only the minimum image can be in range
      d[u] -= a.L[u] * rint(d[u] * a.invL[u]);
      lo[u] = hi[u] = 0;
    } else {
      lo[u] = (int)ceil((-a.rc - d[u]) * a.invL[u]);
      hi[u] = (int)floor((a.rc - d[u]) * a.invL[u]);
    }
  }
  double acc = 0.0;
  for (int i = lo[0]; i <= hi[0]; ++i) {
    const double x = d[0] + i * a.L[0];
    for (int j = lo[1]; j <= hi[1]; ++j) {
      const double y = d[1] + j * a.L[1];
      const double xy = x * x + y * y;
      if (xy >= a.rc2) continue;
      for (int k = lo[2]; k <= hi[2]; ++k) {
        const double z = d[2] + k * a.L[2];
        const double r2 = xy + z * z;
        if (r2 >= a.rc2 || r2 == 0.0) continue;
        const double r = sqrt(r2);
        double e = erfc(a.g * r);
        // erfc(6) < 3e-17: beyond alpha r = 6 the Gaussian term is below double rounding
        // of the erfc(g r) term
        if (ai * r < 6.0) e -= erfc(ai * r);
        acc += q * e / r;
      }
    }
  }
  return acc;
}

// kPool: far terms go to the pool (float storage, listed images).  Blocks an SM: three, where the
// nearest image is all: in the 64 registers of a fourth the compiler leaves less of a warp's work
// in flight, and grids of two or three blocks an SM are slower by up to 15% (12,094 atoms, 8 frames
// of 4,000 ions 1,645 us a call, 1,434 so; many waves gain 1%).  Four for lists of shifts (512
// atoms, 256 frames: 5,394 us a call with three, 5,186 so), but three with the pool, whose
// grids are small.
template <int kMode, bool kF64, bool kPool>
__global__ void __launch_bounds__(kRealWarps * 32, kMode == kShiftList && !kPool ? 4 : 3)
k_bsol_real(const __grid_constant__ RealArgs a) {
  constexpr int kBits = kIonBits<kMode>;
  constexpr bool kFar = !kF64;  // far images apart
  // a lane's near pairs from the start of its list and its far ones from the end, and the 32
  // ions of a step that the bounding box lets through
  __shared__ uint16_t list[kRealWarps][kListDepth][32];
  __shared__ float4 cand[kMode == kSingleImage ? kRealWarps : 1][32];
  __shared__ double red[kRealWarps][32];
  const int f = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int per = (blockDim.x >> 5) / a.shares;  // groups of 32 atoms a block
  const int grp = blockIdx.x * per + warp / a.shares;
  const int i = grp * 32 + lane;
  const bool live = i < a.n;
  wait_previous();
  const IonRec* ions = fresh(a.ions) + (size_t)f * a.n_ion;
  uint32_t ui[3] = {0, 0, 0};
  AtomRec at = {};
  double ri[3] = {0.0, 0.0, 0.0}, ai = 0.0;
  if (live) {
    for (int u = 0; u < 3; ++u) ui[u] = a.sfix[3 * i + u];
    if constexpr (kF64) {
      for (int u = 0; u < 3; ++u) ri[u] = a.xyz[3 * i + u];
    } else {
      at = a.atoms[i];
    }
    ai = a.alpha[i];
  }
  // bounding box of the warp's atoms around a centre, and each atom's offset from it
  uint32_t centre[3];
  float half[3], off[3];
  bool wrap = false;  // an ion in range could lie across the box edge from the centre
  if constexpr (kMode == kSingleImage) {
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      const uint32_t u0 = __shfl_sync(0xffffffffu, ui[u], 0);  // lane 0 is live if any is
      const int d = live ? (int32_t)(ui[u] - u0) : 0;
      const int lo = __reduce_min_sync(0xffffffffu, d), hi = __reduce_max_sync(0xffffffffu, d);
      const long long ext = (long long)hi - lo;
      centre[u] = u0 + (uint32_t)(lo + (int32_t)(ext >> 1));
      half[u] = 0.5f * (float)ext * a.fs[u] + 1e-3f;
      off[u] = (float)(int32_t)(ui[u] - centre[u]) * a.fs[u];
      wrap |= half[u] > a.reach[u];
    }
  }
  float acch = 0.f, accl = 0.f, accf = 0.f;
  const int sh = blockIdx.z * a.shares + warp % a.shares;
  const size_t row = ((size_t)sh * gridDim.y + f) * ((a.n + 31) / 32) + grp;
  int* mine = a.far_row + row * a.far_len;
  float* far = nullptr;  // where this lane's next far term goes
  int nfar = 0, have = 0;  // far terms of the lane, blocks of the warp
  double acc = 0.0;
  int cn = 0, cf = 0;  // near and far entries of this lane's list
  int base0 = 0;
  // far images of this lane's atom: beyond alpha r = 6 as well
  const float lane_far2 = kFar ? fmaxf(a.far2, 36.0f / ((float)(ai * ai))) : 0.f;

  // lists the image of ion t at r^2 = m2 by the screen's float, if it is in range
  auto put = [&](float m2, uint32_t entry) {
    if (!live || m2 >= a.screen2) return;
    if (kFar && m2 >= lane_far2 && m2 < a.cut2) list[warp][kListDepth - ++cf][lane] = (uint16_t)entry;
    else list[warp][cn++][lane] = (uint16_t)entry;
  };

  auto evaluate = [&](uint32_t entry) {
    const int ion = base0 + (int)(entry & ((1u << kBits) - 1));
    const int si = kMode == kShiftList ? (int)(entry >> kBits) : 0;
    if constexpr (kF64 || kMode == kAllImages) {
      const size_t e = (size_t)f * a.n_ion + ion;
      const double p[3] = {a.ion_xyz[3 * e], a.ion_xyz[3 * e + 1], a.ion_xyz[3 * e + 2]};
      if constexpr (kMode == kAllImages) {
        const double rr[3] = {a.xyz[3 * i], a.xyz[3 * i + 1], a.xyz[3 * i + 2]};
        acc += pair_images(rr, ai, p, a.ion_q[e], a);
      } else {
        // the image: the fixed-point nearest one (whole boxes k from the FP64 difference)
        // plus the listed shift
        const uint32_t uI[3] = {ions[ion].x, ions[ion].y, ions[ion].z};
        double r2 = 0.0;
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          const double dd = ri[u] - p[u];
          const double dfx = (double)(int32_t)(ui[u] - uI[u]) * (a.L[u] * 0x1p-32);
          double k = rint((dd - dfx) * a.invL[u]);
          if constexpr (kMode == kShiftList) k -= (double)a.kshift[si][u];
          const double du = dd - k * a.L[u];
          r2 += du * du;
        }
        if (r2 < a.rc2 && r2 > 0.0) {
          const double r = sqrt(r2);
          double e2 = erfc(a.g * r);
          if (ai * r < 6.0) e2 -= erfc(ai * r);
          acc += a.ion_q[e] * e2 / r;
        }
      }
    } else {
      const uint4 w0 = __ldca(reinterpret_cast<const uint4*>(ions + ion));
      const int4 w1 = __ldca(reinterpret_cast<const int4*>(ions + ion) + 1);
      const uint32_t uI[3] = {w0.x, w0.y, w0.z};
      const int32_t lI[3] = {w1.x, w1.y, w1.z};
      const int32_t la[3] = {at.xl, at.yl, at.zl};
      float sh = 0.f, sl = 0.f;  // r^2
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        // the difference in units of 2^-32 box: top 24 bits exact as a float, then the rest
        const int32_t d = (int32_t)(ui[u] - uI[u]);
        float dh = (float)(d & ~0xFF);
        float dl = (float)(d & 0xFF) + ((float)la[u] - (float)lI[u]) * 0x1p-32f;
        if constexpr (kMode == kShiftList) {
          // whole boxes: 2^32 k units, a two-sum
          const float k = (float)a.kshift[si][u] * 4294967296.0f;
          const float s = dh + k, bb = s - dh;
          dl += (dh - (s - bb)) + (k - bb);
          dh = s;
        }
        float xh, xl;
        ff_mul(dh, dl, a.fsh[u], a.fsl[u], xh, xl);
        const float p = __fmul_rn(xh, xh);
        pair_add_pair(sh, sl, p, fmaf(xh, xh, -p) + 2.0f * xh * xl);
      }
      // strictly inside r_c
      if ((sh - a.rc2h) + (sl - a.rc2l) < 0.f) {
        float gh, gl, bh, bl, vh, vl;
        ff_mul(sh, sl, a.g2h, a.g2l, gh, gl);
        ff_mul(sh, sl, at.ah, at.al, bh, bl);
        if (fminf(gh, bh) >= kHMin) {
          // q g [H(g^2 r^2) - (alpha / g) H(alpha^2 r^2)]; beyond alpha r = 6 the second
          // term is below 1e-17 of the first
          vh = vl = 0.f;
          if (gh < 64.0f) h_table(a.htab, gh, gl, vh, vl);
          if (bh < 36.0f) {
            float hh, hl;
            h_table(a.htab, bh, bl, hh, hl);
            float ph, pl;
            ff_mul(hh, hl, at.bh, at.bl, ph, pl);
            ff_add(vh, vl, ph, pl, vh, vl);
          }
          float ph, pl;
          ff_mul(vh, vl, a.gh, a.gl, ph, pl);
          ff_mul(ph, pl, __uint_as_float(w0.w), __int_as_float(w1.w), vh, vl);
          pair_add_pair(acch, accl, vh, vl);
        } else {  // an ion almost on an atom: FP64
          const double r2 = (double)sh + (double)sl;
          if (r2 > 0.0) {
            const double r = sqrt(r2);
            double e2 = erfc(a.g * r);
            if (ai * r < 6.0) e2 -= erfc(ai * r);
            acc += a.ion_q[(size_t)f * a.n_ion + ion] * e2 / r;
          }
        }
      }
    }
  };
  // a far image, in plain float from the fixed-point difference of the nearest image; one
  // that the screen's offsets took for far and this r^2 does not goes the near way
  auto evaluate_far = [&](uint32_t entry) {
    const uint4 w = __ldca(reinterpret_cast<const uint4*>(ions + base0 + (entry & ((1u << kBits) - 1))));
    float d0 = (float)(int32_t)(ui[0] - w.x) * a.fs[0], d1 = (float)(int32_t)(ui[1] - w.y) * a.fs[1],
          d2 = (float)(int32_t)(ui[2] - w.z) * a.fs[2];
    float m2;
    if constexpr (kMode == kShiftList) {
      const int si = (int)(entry >> kBits);
      d0 += a.shift[si][0];
      d1 += a.shift[si][1];
      d2 += a.shift[si][2];
      m2 = fmaf(d2, d2, fmaf(d1, d1, d0 * d0));
    } else {
      m2 = fmaf(d0, d0, fmaf(d1, d1, d2 * d2));
    }
    if (m2 >= lane_far2 && m2 < a.cut2) {
      const float ir = rsqrtf(m2);  // 1 / r to ~2 ulp
      const float q = __uint_as_float(w.w), e = erfcf(a.gh * (m2 * ir)) * ir;
      if constexpr (kPool) {
        if (nfar % kFarTerms == 0)
          far = a.far + (size_t)mine[nfar / kFarTerms] * (kFarTerms * 32) + lane;
        *far = q * e;
        far += 32;
        ++nfar;
      } else {
        accf += q * e;
      }
    } else {
      evaluate(entry);
    }
  };
  // evaluates every listed pair of the warp
  auto drain = [&]() {
    int most = __reduce_max_sync(0xffffffffu, cn);
    for (int k = 0; k < most; ++k)
      if (k < cn) evaluate(list[warp][k][lane]);
    cn = 0;
    if constexpr (kFar) {
      if constexpr (kPool) {  // blocks for what is listed
        const int more = (__reduce_max_sync(0xffffffffu, nfar + cf) + kFarTerms - 1) / kFarTerms -
                         have;
        if (more > 0) {
          unsigned b = 0;
          if (lane == 0) {
            b = atomicAdd(a.far_state, (unsigned)more);
            if (b + more > (unsigned)a.far_blocks) {
              a.far_state[1] = 1u;
              b = ~0u;
            }
          }
          b = __shfl_sync(0xffffffffu, b, 0);
          for (int k = lane; k < more; k += 32) mine[have + k] = b == ~0u ? 0 : (int)b + k;
          have += more;
          __syncwarp();
        }
      }
      most = __reduce_max_sync(0xffffffffu, cf);
      for (int k = 1; k <= most; ++k)
        if (k <= cf) evaluate_far(list[warp][kListDepth - k][lane]);
      cf = 0;
    }
  };

  // this warp's share of the ions
  const int nsh = a.shares * gridDim.z;
  const int t0 = (int)((int64_t)a.n_ion * sh / nsh), t1 = (int)((int64_t)a.n_ion * (sh + 1) / nsh);
  base0 = t0;
  int since = 0;  // screened since the lists were last looked at
  auto look = [&](int steps) {  // before screening `steps` (at most kListStep) more
    if (since + steps > kListStep) {
      since = 0;
      if (__any_sync(0xffffffffu, cn + cf >= kListDepth - kListStep)) drain();
    }
    since += steps;
  };
  if (grp * 32 < a.n)
    for (int t = t0; t < t1; t += 32) {
      if (t - base0 > (1 << kBits) - 32) {  // the entries' range of ions
        drain();
        base0 = t;
      }
      const int m = min(32, t1 - t);
      if constexpr (kMode == kSingleImage) {
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        bool in = lane < m;
        float dx[3];
        if (in) w = __ldca(reinterpret_cast<const uint4*>(ions + t + lane));
        const uint32_t uI[3] = {w.x, w.y, w.z};
        float far2 = 0.f;
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          dx[u] = (float)(int32_t)(uI[u] - centre[u]) * a.fs[u];
          const float e = fmaxf(fabsf(dx[u]) - half[u], 0.f);
          far2 = fmaf(e, e, far2);
        }
        in = in && far2 < a.screen2;
        const unsigned mask = __ballot_sync(0xffffffffu, in);
        const int k = __popc(mask);
        if (!k) continue;
        __syncwarp();  // the last step's reads of cand are done
        if (in) {
          const int p = __popc(mask & ((1u << lane) - 1u));
          // offsets from the centre, or (an ion could lie across the box edge) the
          // fixed-point coordinates themselves
          cand[warp][p] = wrap ? make_float4(__uint_as_float(w.x), __uint_as_float(w.y),
                                             __uint_as_float(w.z), __int_as_float(t + lane))
                               : make_float4(dx[0], dx[1], dx[2], __int_as_float(t + lane));
        }
        __syncwarp();
        for (int c0 = 0; c0 < k; c0 += kListStep) {
          const int c1 = min(k, c0 + kListStep);
          look(c1 - c0);
#pragma unroll 2
          for (int c = c0; c < c1; ++c) {
            const float4 p = cand[warp][c];
            float x, y, z;
            if (wrap) {
              x = (float)(int32_t)(ui[0] - __float_as_uint(p.x)) * a.fs[0];
              y = (float)(int32_t)(ui[1] - __float_as_uint(p.y)) * a.fs[1];
              z = (float)(int32_t)(ui[2] - __float_as_uint(p.z)) * a.fs[2];
            } else {
              x = off[0] - p.x;
              y = off[1] - p.y;
              z = off[2] - p.z;
            }
            put(fmaf(x, x, fmaf(y, y, z * z)), (uint32_t)(__float_as_int(p.w) - base0));
          }
        }
      } else {
        for (int c = 0; c < m; ++c) {
          const uint4 w = __ldca(reinterpret_cast<const uint4*>(ions + t + c));
          const float x = (float)(int32_t)(ui[0] - w.x) * a.fs[0];
          const float y = (float)(int32_t)(ui[1] - w.y) * a.fs[1];
          const float z = (float)(int32_t)(ui[2] - w.z) * a.fs[2];
          if constexpr (kMode == kAllImages) {
            look(1);
            put(fmaf(x, x, fmaf(y, y, z * z)), (uint32_t)(t + c - base0));
          } else {
            for (int s0 = 0; s0 < a.nshift; s0 += kListStep) {
              const int s1 = min(a.nshift, s0 + kListStep);
              look(s1 - s0);
              for (int si = s0; si < s1; ++si) {
                const float sx = x + a.shift[si][0], sy = y + a.shift[si][1],
                            sz = z + a.shift[si][2];
                put(fmaf(sz, sz, fmaf(sy, sy, sx * sx)),
                    ((uint32_t)si << kBits) | (uint32_t)(t + c - base0));
              }
            }
          }
        }
      }
    }
  drain();
  acc += (double)accf;
  acc += (double)acch + (double)accl;
  if (kPool && live) a.far_count[row * 32 + lane] = nfar;
  if (a.shares > 1) {  // the block's shares of a group, in share order
    red[warp][lane] = acc;
    __syncthreads();
    if (warp % a.shares != 0) return;
    for (int s = 1; s < a.shares; ++s) acc += red[warp + s][lane];
  }
  if (live) a.part[((size_t)blockIdx.z * gridDim.y + f) * a.n + i] = acc;
}

struct FinishArgs {
  const double* part;  // [shares][frames][n] real-space sums
  int shares, n;
  const float* far;  // far terms of the shares (far_blocks 0: none)
  const unsigned* far_state;
  const int *far_row, *far_count;
  int far_shares, far_blocks, far_len;
  const double2* sums;  // [frames][nsum] (sum q z, sum q)
  int nsum;
  const double* xyz;
  double dip;  // 4 pi / V in slab geometry
  const double *chi, *bsol_k;
  double *b_out, *qsol;
  unsigned long long* stamp;  // start and end
  unsigned long long* over;   // whether the far terms outgrew their pool
};

// b = chi - k_e (b^sol_k + real + dipole term), the real-space shares in share order; every warp
// adds the frame's block sums.
__global__ void __launch_bounds__(128) k_bsol_finish(const __grid_constant__ FinishArgs a) {
  wait_previous();
  stamp_time(a.stamp);
  const int f = blockIdx.y, i = blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const double* part = fresh(a.part);
  const double2* sums = fresh(a.sums);
  const double* bsol_k = fresh(a.bsol_k);
  double real = 0.0;
  if (i < a.n)
    for (int z = 0; z < a.shares; ++z) real += part[((size_t)z * gridDim.y + f) * a.n + i];
  if (a.far_blocks > 0 && i < a.n) {  // one float chain over the shares, as one warp adds them
    const float* far = fresh(a.far) + lane;
    const int *rows = fresh(a.far_row), *count = fresh(a.far_count);
    float c = 0.f;
    for (int z = 0; z < a.far_shares; ++z) {
      const size_t row = ((size_t)z * gridDim.y + f) * ((a.n + 31) / 32) + (i >> 5);
      const int m = count[row * 32 + lane];
      for (int k0 = 0; k0 < m; k0 += kFarTerms) {
        const float* t =
            far + (size_t)rows[row * a.far_len + k0 / kFarTerms] * (kFarTerms * 32);
        float x[kFarTerms];
#pragma unroll
        for (int k = 0; k < kFarTerms; ++k) x[k] = k0 + k < m ? t[k * 32] : 0.f;
#pragma unroll
        for (int k = 0; k < kFarTerms; ++k)
          if (k0 + k < m) c += x[k];
      }
    }
    real += (double)c;
    if (a.over && i == 0 && f == 0) *a.over = fresh(a.far_state)[1];
  }
  double qz = 0.0, qs = 0.0;
  for (int s = lane; s < a.nsum; s += 32) {
    const double2 v = sums[(size_t)f * a.nsum + s];
    qz += v.x;
    qs += v.y;
  }
  for (int o = 16; o; o >>= 1) {
    qz += __shfl_xor_sync(0xffffffffu, qz, o);
    qs += __shfl_xor_sync(0xffffffffu, qs, o);
  }
  if (i < a.n) {
    const size_t e = (size_t)f * a.n + i;
    const double bs = bsol_k[e] + real + a.dip * a.xyz[3 * i + 2] * qz;
    a.b_out[e] = a.chi[i] - kKe * bs;
  }
  if (i == 0 && a.qsol) a.qsol[f] = qs;
  if (a.stamp && blockIdx.x == gridDim.x - 1 && blockIdx.y == gridDim.y - 1 && threadIdx.x == 0)
    a.stamp[1] = now_ns();
}

int prep_blocks(int n_ion) { return (n_ion + kPrepThreads - 1) / kPrepThreads; }

// Shifts k with |k| <= m = floor((r_c + L / 2) / L) per direction (only k = 0 where L > 2 r_c):
// every image within r_c of an atom, given the nearest one.  list: they fit the screen's.
struct Shifts {
  int m[3], total;
  bool all_single, list;
};

Shifts whole_box_shifts(const Geometry& geo) {
  Shifts sh;
  sh.total = 1;
  sh.all_single = true;
  for (int u = 0; u < 3; ++u) {
    const bool single = 2.0 * geo.rc < geo.L[u];
    sh.all_single &= single;
    sh.m[u] = single ? 0 : (int)floor((geo.rc + 0.5 * geo.L[u]) / geo.L[u]);
    sh.total *= 2 * sh.m[u] + 1;
  }
  sh.list = sh.total <= kMaxShifts;
  return sh;
}

}  // namespace

size_t h_table_bytes() { return 8 * kHIntervals * sizeof(float); }

const void* h_table_host() {
  static const std::vector<float> tab = make_h_table();  // once per process
  return tab.data();
}

size_t atom_record_bytes(int n) { return (size_t)n * sizeof(AtomRec); }

void launch_atom_records(const double* xyz, const double* alpha, int n, const Geometry& geo,
                         void* rec, cudaStream_t s) {
  (k_atom_records<<<(n + 127) / 128, 128, 0, s>>>(xyz, alpha, n, geo.L[0], geo.L[1], geo.L[2],
                                                  geo.g, (AtomRec*)rec), note_launch());
}

// Scratch of the real-space part: ion records, block sums, and the grid shares' partials.
// Warps of a block split the ions of one group of atoms until the chip's warps are busy (24
// resident an SM); where eight shares leave SMs without a block, the grid splits them
// further: shares of at least 32 ions, the step of a warp, or, where the images of every ion
// are screened one by one (a box edge below 2 r_c), of eight (512 atoms, 200 ions: 18.9 us
// in 16 blocks, 9.2 in 48).
// Float storage adds an atom's far images in one float chain, in the ions' order; its rounding is
// most of the real-space error where the ions are many (1e-9 of b at 5,000 ions in a small box),
// and sums by shares would exchange it for another, so that b would move by as much with the
// number of frames.  Above kRealChainIons the shares therefore leave their far terms in scratch
// and the finish adds them in order.  The warps take blocks of 16 terms a lane from one pool
// as their lists grow: ions that are sorted in space give one share most of an atom's terms,
// but not more of them (lists of a fixed length a share overflowed there, and the rest of the terms
// was summed by the share).  The pool holds four times the mean number of images within r_c of
// an atom (ions fill part of the box) and a block a warp.  Where that takes more than kRealFarBytes
// the ions stay together, in blocks of fewer warps, and where a pool was too small after all
// (ions in a small part of the box, and atoms in no order, so that every warp has a lane with all of
// them) the caller sums them again that way.  One frame of 2,000 ions, 320 atoms: 170 us a call
// (209 with lists of a fixed length, 110 with sums by shares, 1,800 with the ions together); 5,341
// atoms, 5,000 ions, two frames: 750 (963, 767, 1,958).
constexpr int kRealChainIons = 1200;
constexpr size_t kRealFarBytes = (size_t)192 << 20;

RealPlan real_plan(int n, int frames, int n_ion, const Geometry& geo, bool fp64, int sms,
                   bool small) {
  RealPlan p;
  const int64_t groups = (int64_t)((n + 31) / 32) * frames;
  p.shares = p.grid_shares = 1;
  p.warps = kRealWarps;
  p.far_blocks = p.far_row = 0;
  while (p.shares < kRealWarps && groups * p.shares < 24 * (int64_t)sms) p.shares *= 2;
  const int64_t blocks = (groups * p.shares + kRealWarps - 1) / kRealWarps;
  const Shifts sh = whole_box_shifts(geo);
  p.grid_shares = (int)std::max<int64_t>(
      1, std::min<int64_t>((sms + blocks - 1) / blocks,
                           n_ion / ((sh.all_single ? 32 : 8) * p.shares)));
  // (every image of a pair goes to FP64 sums where the shifts are not listed)
  if (!fp64 && sh.list && n_ion > kRealChainIons && p.shares * p.grid_shares > 1) {
    const int nsh = p.shares * p.grid_shares;
    const double mean = n_ion * (4.0 / 3.0 * kPi * geo.rc * geo.rc * geo.rc) /
                        (geo.L[0] * geo.L[1] * geo.L[2]);
    const double rows = (double)groups * nsh;
    const int len = ((n_ion + nsh - 1) / nsh * sh.total + kFarTerms - 1) / kFarTerms;
    const double pool = std::min(rows * len, rows * (4.0 * mean / nsh / kFarTerms + 1.0));
    if (!small && pool * kFarTerms * 32 * sizeof(float) + rows * len * sizeof(int) <=
                      (double)kRealFarBytes) {
      p.far_blocks = (int)pool;
      p.far_row = len;
    } else {
      p.shares = p.grid_shares = 1;
      p.warps =
          (int)std::max<int64_t>(1, std::min<int64_t>(kRealWarps, groups / (2 * (int64_t)sms)));
    }
  }
  auto up = [](size_t b) { return (b + 255) & ~size_t(255); };
  p.o_sums = up((size_t)frames * std::max(n_ion, 1) * sizeof(IonRec));
  p.o_part = p.o_sums + up((size_t)frames * std::max(prep_blocks(n_ion), 1) * sizeof(double2));
  p.o_far = p.o_part + up((size_t)p.grid_shares * frames * n * sizeof(double));
  const size_t rows = (size_t)p.shares * p.grid_shares * groups;
  p.o_far_state = p.o_far + up((size_t)p.far_blocks * kFarTerms * 32 * sizeof(float));
  p.o_far_row = p.o_far_state + (p.far_blocks > 0 ? 256 : 0);
  p.o_far_count = p.o_far_row + up(rows * p.far_row * sizeof(int));
  p.bytes = p.o_far_count + (p.far_blocks > 0 ? up(rows * 32 * sizeof(int)) : 0);
  return p;
}

void launch_ion_prepare(const double* ion_xyz, const double* ion_q, int frames, int n_ion,
                        const Geometry& geo, uint32_t* sion, const RealPlan& plan, void* scratch,
                        unsigned long long* stamp, cudaStream_t s) {
  (k_ion_prepare<<<dim3(prep_blocks(n_ion), frames), kPrepThreads, 0, s>>>(
       ion_xyz, ion_q, n_ion, geo.L[0], geo.L[1], geo.L[2], sion, (IonRec*)scratch,
       (double2*)((char*)scratch + plan.o_sums),
       plan.far_blocks > 0 ? (unsigned*)((char*)scratch + plan.o_far_state) : nullptr, stamp),
   note_launch());
}

// Launched after the ions' preparation, which it waits for; what comes after may start beside it.
void launch_bsol_real(const double* xyz, const double* alpha, const uint32_t* sfix,
                      const void* atoms, const void* htab, int n, const double* ion_xyz,
                      const double* ion_q, int frames, int n_ion, const Geometry& geo, bool fp64,
                      const RealPlan& plan, void* scratch, cudaStream_t s) {
  RealArgs a;
  a.xyz = xyz;
  a.alpha = alpha;
  a.sfix = sfix;
  a.atoms = (const AtomRec*)atoms;
  a.n = n;
  a.ion_xyz = ion_xyz;
  a.ion_q = ion_q;
  a.ions = (const IonRec*)scratch;
  a.n_ion = n_ion;
  a.shares = plan.shares;
  a.htab = (const float4*)htab;
  a.g = geo.g;
  a.rc = geo.rc;
  a.rc2 = geo.rc * geo.rc;
  a.screen2 = (float)a.rc2 + 0.01f;
  auto pair = [](double v, float& h, float& l) {
    h = (float)v;
    l = (float)(v - (double)h);
  };
  pair(a.rc2, a.rc2h, a.rc2l);
  pair(geo.g * geo.g, a.g2h, a.g2l);
  pair(geo.g, a.gh, a.gl);
  // r_split: erfc(g r) / r = 1e-4 / A (bisection); r_c (no far images) where the term never
  // gets that small
  double lo = 1e-3, hi = geo.rc;
  if (erfc(geo.g * hi) / hi <= 1e-4)
    for (int it = 0; it < 60; ++it) {
      const double mid = 0.5 * (lo + hi);
      if (erfc(geo.g * mid) / mid > 1e-4) lo = mid;
      else hi = mid;
    }
  a.far2 = (float)(hi * hi);
  a.cut2 = (float)(a.rc2 * (1.0 - 1e-5));
  for (int u = 0; u < 3; ++u) {
    a.L[u] = geo.L[u];
    a.invL[u] = 1.0 / geo.L[u];
    a.single[u] = 2.0 * geo.rc < geo.L[u];
    a.fs[u] = (float)(geo.L[u] * 0x1p-32);
    pair(geo.L[u] * 0x1p-32, a.fsh[u], a.fsl[u]);
    a.reach[u] = (float)(0.5 * geo.L[u] - geo.rc) - 0.01f;
  }
  const Shifts sh = whole_box_shifts(geo);
  const int* m = sh.m;
  a.nshift = sh.list ? sh.total : 0;
  int k = 0;
  for (int x = -m[0]; a.nshift && x <= m[0]; ++x)
    for (int y = -m[1]; y <= m[1]; ++y)
      for (int z = -m[2]; z <= m[2]; ++z, ++k) {
        const int ks[3] = {x, y, z};
        for (int u = 0; u < 3; ++u) {
          a.shift[k][u] = (float)(ks[u] * geo.L[u]);
          a.kshift[k][u] = (signed char)ks[u];
        }
      }
  a.part = (double*)((char*)scratch + plan.o_part);
  a.far = (float*)((char*)scratch + plan.o_far);
  a.far_state = (unsigned*)((char*)scratch + plan.o_far_state);
  a.far_row = (int*)((char*)scratch + plan.o_far_row);
  a.far_count = (int*)((char*)scratch + plan.o_far_count);
  a.far_blocks = plan.far_blocks;
  a.far_len = plan.far_row;
  const int groups = (n + 31) / 32, per = plan.warps / plan.shares;
  const dim3 grid((groups + per - 1) / per, frames, plan.grid_shares);
  const bool pool = plan.far_blocks > 0;
  auto kernel = sh.all_single ? (fp64   ? k_bsol_real<kSingleImage, true, false>
                                 : pool ? k_bsol_real<kSingleImage, false, true>
                                        : k_bsol_real<kSingleImage, false, false>)
                : sh.list     ? (fp64   ? k_bsol_real<kShiftList, true, false>
                                 : pool ? k_bsol_real<kShiftList, false, true>
                                        : k_bsol_real<kShiftList, false, false>)
                              : k_bsol_real<kAllImages, true, false>;
  launch_next(kernel, grid, plan.warps * 32, 0, s, a);
}

void launch_bsol_finish(const double* xyz, int n, int frames, int n_ion, const Geometry& geo,
                        const double* chi, const double* bsol_k, double* b_out, double* qsol,
                        const RealPlan& plan, void* scratch, unsigned long long* stamp,
                        unsigned long long* over, cudaStream_t s) {
  FinishArgs a;
  a.part = (const double*)((char*)scratch + plan.o_part);
  a.shares = plan.grid_shares;
  a.far = (const float*)((char*)scratch + plan.o_far);
  a.far_state = (const unsigned*)((char*)scratch + plan.o_far_state);
  a.far_row = (const int*)((char*)scratch + plan.o_far_row);
  a.far_count = (const int*)((char*)scratch + plan.o_far_count);
  a.far_shares = plan.shares * plan.grid_shares;
  a.far_blocks = plan.far_blocks;
  a.far_len = plan.far_row;
  a.over = over;
  a.n = n;
  a.sums = (const double2*)((char*)scratch + plan.o_sums);
  a.nsum = prep_blocks(n_ion);
  a.xyz = xyz;
  a.dip = geo.slab ? 4.0 * kPi / geo.vol : 0.0;
  a.chi = chi;
  a.bsol_k = bsol_k;
  a.b_out = b_out;
  a.qsol = qsol;
  a.stamp = stamp;
  launch_next(k_bsol_finish, dim3((n + 127) / 128, frames), 128, 0, s, a);
}

}  // namespace cpm
