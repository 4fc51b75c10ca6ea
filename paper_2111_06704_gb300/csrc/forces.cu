// Forces on the ions from the electrode charges: F_I = -q_I d/dr_I sum_i q_i e_iI (Eq. S25
// inside the Ewald sums of Eq. 22 / 25, the paper's form with Eq. 39).
//
// Reciprocal part: d/dr_I cos(K.(r_i - r_I)) = sin(K.(r_i - r_I)) K, so with the
// electrode's charge-weighted structure factors (C_K, S_K) = sum_i q_i (cos, sin)(K.r_i),
// grad_I = sum_K W_K [S_K cos(K.r_I) - C_K sin(K.r_I)] K.  v holds sqrt(W) (C, S) in the
// operand's column layout (the ions' structure-factor kernel run over the electrode), so
// the term is sqrt(W_K) (v_s cos - v_c sin); the integer h, k, l multiply last:
// K = 2 pi (h/Lx, k/Ly, l/Lz).
//
// An MD step has few ions (hundreds to thousands) against up to 10^5 k-vectors and
// electrode atoms, so both parts split the long sum over the grid as well as the ions; the
// shares go to scratch and k_force_finish adds them in a fixed order.
#include <math.h>

#include <algorithm>

#include "phasor.cuh"
#include "programmatic.cuh"

namespace cpm {

namespace {

constexpr int kFkIons = 8;       // ions a block of the k-space kernels
constexpr int kFkThreads = 128;  // k-vectors in flight a block

// Sums the threads' float-pair gradients (8 ions x 3 components) over the block and writes
// them in FP64.
__device__ __forceinline__ void write_gradients(float2 (&gh)[kFkIons / 2][3],
                                                float2 (&gl)[kFkIons / 2][3], int i0, int n_ion,
                                                double* __restrict__ out) {
  __shared__ float2 red[kFkThreads / 32][kFkIons * 3];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int u = 0; u < kFkIons; ++u)
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      float h = (u & 1) ? gh[u >> 1][d].y : gh[u >> 1][d].x;
      float l = (u & 1) ? gl[u >> 1][d].y : gl[u >> 1][d].x;
#pragma unroll
      for (int o = 16; o; o >>= 1)
        pair_add_pair(h, l, __shfl_xor_sync(0xffffffffu, h, o),
                      __shfl_xor_sync(0xffffffffu, l, o));
      if (lane == 0) red[warp][u * 3 + d] = make_float2(h, l);
    }
  __syncthreads();
  if (threadIdx.x < kFkIons * 3 && i0 + (int)threadIdx.x / 3 < n_ion) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kFkThreads / 32; ++w) {
      const float2 e = red[w][threadIdx.x];
      s += (double)e.x + (double)e.y;
    }
    out[3 * (size_t)i0 + threadIdx.x] = s;
  }
}

// Float storage: gradient shares of 8 ions over one share of the k range, part[share][frame]
// [ion][3].  A thread takes every 128th k-vector of the share for all 8 ions, so a
// k-vector's index, weight and structure factors are read once for 8 phasors, and the ions
// go in pairs through paired float instructions.  Shares 0 .. nsplit - 1 hold the tail
// k-vectors (float phasors from the table, one ulp, each term times h, k, l unrounded into a
// float pair); share nsplit, where there is one, the head (k < kh, the heaviest weights) in float
// pairs throughout (~1e-13: FP64 runs at 1/64 of the float rate).  One thread per ion over
// the whole k range, the form before, kept 16 blocks of the chip busy with 2,000 ions:
// 30.7 ms with 217,619 k-vectors against 0.83 ms.
__global__ void __launch_bounds__(kFkThreads)
k_force_kspace(const uint32_t* __restrict__ sion, int n_ion, const int* __restrict__ hkl,
               const double* __restrict__ sqw, int mpad, int kh, int nsplit,
               const float4* __restrict__ turn, const float* __restrict__ v,
               const float2* __restrict__ vhead, double* __restrict__ part) {
  wait_previous(false);
  sion = fresh(sion);
  v = fresh(v);
  vhead = fresh(vhead);
  const int f = blockIdx.y, frames = gridDim.y, sp = blockIdx.z;
  const int i0 = blockIdx.x * kFkIons;
  uint32_t u[kFkIons][3];
#pragma unroll
  for (int t = 0; t < kFkIons; ++t) {  // an ion past the last repeats it and is not written
    const uint32_t* p = sion + ((size_t)f * n_ion + min(i0 + t, n_ion - 1)) * 3;
#pragma unroll
    for (int d = 0; d < 3; ++d) u[t][d] = __ldca(p + d);
  }
  float2 gh[kFkIons / 2][3], gl[kFkIons / 2][3];
#pragma unroll
  for (int p = 0; p < kFkIons / 2; ++p)
#pragma unroll
    for (int d = 0; d < 3; ++d) gh[p][d] = gl[p][d] = make_float2(0.f, 0.f);
  if (sp < nsplit) {
    const int64_t tail = mpad - kh;
    const int k1 = kh + (int)(tail * (sp + 1) / nsplit);
    const float* vf = v + (size_t)f * 2 * mpad;
    for (int k = kh + (int)(tail * sp / nsplit) + threadIdx.x; k < k1; k += kFkThreads) {
      const uint32_t h0 = (uint32_t)hkl[3 * k], h1 = (uint32_t)hkl[3 * k + 1],
                     h2 = (uint32_t)hkl[3 * k + 2];
      const size_t kcol = 128 * (size_t)(k >> 6) + (k & 63);
      const float w = (float)sqw[k], vc = vf[kcol], vs = vf[kcol + 64];
      // h, k, l: small integers, exact as floats
      const float hf[3] = {(float)(int)h0, (float)(int)h1, (float)(int)h2};
#pragma unroll
      for (int p = 0; p < kFkIons / 2; ++p) {
        float2 sn, cs;
        sincos_table(h0 * u[2 * p][0] + h1 * u[2 * p][1] + h2 * u[2 * p][2], turn, &sn.x, &cs.x);
        sincos_table(h0 * u[2 * p + 1][0] + h1 * u[2 * p + 1][1] + h2 * u[2 * p + 1][2], turn,
                     &sn.y, &cs.y);
        const float2 term =
            __fmul2_rn(make_float2(w, w), __ffma2_rn(make_float2(vs, vs), cs,
                                                     __fmul2_rn(make_float2(-vc, -vc), sn)));
#pragma unroll
        for (int d = 0; d < 3; ++d)
          pair_fma2(gh[p][d], gl[p][d], term, make_float2(hf[d], hf[d]));
      }
    }
  } else {
    const float2* vh = vhead + (size_t)f * 2 * kh;
    for (int k = threadIdx.x; k < kh; k += kFkThreads) {
      const uint32_t h0 = (uint32_t)hkl[3 * k], h1 = (uint32_t)hkl[3 * k + 1],
                     h2 = (uint32_t)hkl[3 * k + 2];
      const size_t kcol = 128 * (size_t)(k >> 6) + (k & 63);
      const double wd = sqw[k];
      const float wh = (float)wd, wl = (float)(wd - (double)wh);
      const float2 vc = vh[kcol], vs = vh[kcol + 64];
      float ch, cl, sh, sl;
      ff_mul(wh, wl, vc.x, vc.y, ch, cl);
      ff_mul(wh, wl, vs.x, vs.y, sh, sl);
      const float hf[3] = {(float)(int)h0, (float)(int)h1, (float)(int)h2};
#pragma unroll
      for (int t = 0; t < kFkIons; ++t) {
        float cph, cpl, sph, spl, ah, al, bh, bl, th, tl;
        phasor_ff(h0 * u[t][0] + h1 * u[t][1] + h2 * u[t][2], turn, cph, cpl, sph, spl);
        ff_mul(sh, sl, cph, cpl, ah, al);
        ff_mul(ch, cl, sph, spl, bh, bl);
        ff_add(ah, al, -bh, -bl, th, tl);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const float x = __fmul_rn(th, hf[d]);
          const float xl = fmaf(tl, hf[d], fmaf(th, hf[d], -x));
          if (t & 1) pair_add_pair(gh[t >> 1][d].y, gl[t >> 1][d].y, x, xl);
          else pair_add_pair(gh[t >> 1][d].x, gl[t >> 1][d].x, x, xl);
        }
      }
    }
  }
  write_gradients(gh, gl, i0, n_ion, part + ((size_t)sp * frames + f) * n_ion * 3);
}

// FP64 storage: one ion a block, threads over the k-vectors of a share, the phasors as
// products of the ion's per-axis phasors (k_axis_phasors): ten FP64 operations instead of
// a sincospi of some sixty.  part as above.
__global__ void __launch_bounds__(kFkThreads)
k_force_kspace_f64(const double2* __restrict__ axis, AxisPhasors ap, int n_ion,
                   const int* __restrict__ hkl, const double* __restrict__ sqw, int mpad,
                   int nsplit, const double* __restrict__ v, double* __restrict__ part) {
  __shared__ double red[kFkThreads / 32][3];
  wait_previous(false);
  axis = fresh(axis);
  v = fresh(v);
  const int f = blockIdx.y, frames = gridDim.y, sp = blockIdx.z, ion = blockIdx.x;
  const double2* row = axis + ((size_t)f * n_ion + ion) * ap.len;
  const double* vf = v + (size_t)f * 2 * mpad;
  double g[3] = {0.0, 0.0, 0.0};
  const int k1 = (int)((int64_t)mpad * (sp + 1) / nsplit);
  for (int k = (int)((int64_t)mpad * sp / nsplit) + threadIdx.x; k < k1; k += kFkThreads) {
    const int h0 = hkl[3 * k], h1 = hkl[3 * k + 1], h2 = hkl[3 * k + 2];
    const size_t kcol = 128 * (size_t)(k >> 6) + (k & 63);
    const double2 e = ap.phasor(row, h0, h1, h2);
    const double term = sqw[k] * (vf[kcol + 64] * e.x - vf[kcol] * e.y);
    g[0] += term * h0;
    g[1] += term * h1;
    g[2] += term * h2;
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    for (int o = 16; o; o >>= 1) g[d] += __shfl_xor_sync(0xffffffffu, g[d], o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][d] = g[d];
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    double s = 0.0;
    for (int w = 0; w < kFkThreads / 32; ++w) s += red[w][threadIdx.x];
    part[(((size_t)sp * frames + f) * n_ion + ion) * 3 + threadIdx.x] = s;
  }
}

// d/dr [erfc(g r) / r - erfc(a r) / r] (a = INFINITY: a point charge, no Gaussian term).
// Beyond a r = 6.5 the Gaussian term is below 1e-17 of the other.
__device__ __forceinline__ double radial_derivative(double g, double a, double r) {
  const double two_sqrtpi = 1.1283791670955126;  // 2 / sqrt(pi)
  double num = -two_sqrtpi * g * exp(-(g * r) * (g * r));
  double e = erfc(g * r);
  if (a * r < 6.5) {
    num += two_sqrtpi * a * exp(-(a * r) * (a * r));
    e -= erfc(a * r);
  }
  return num / r - e / (r * r);
}

// Real part: gradients of 32 ions (one a lane) over one share of the electrode atoms,
// part[share][frame][ion][3] and the share's slab sums slab[share][frame] = (sum q_i z_i,
// sum q_i).  The block's eight warps take 4 to 32 atoms each of every staged chunk.  A
// pair is screened in float from the exact fixed-point difference of its nearest image
// (0.01 A^2 band, as k_bsol_real); the pairs that pass go to a queue of the warp and are
// summed 32 at a time, all lanes busy, over every image within r_c in FP64:
// grad -= q_i f'(r) / r (r_i - r_I + R); each ion then adds its pairs in queue order.  At
// 2,000 ions and 12,800 atoms 0.4% of the pairs pass, so a lane that evaluated its own
// pairs at once (the form before, one thread an ion, 16 blocks) left the FP64 unit to one
// lane in thirty: 34.6 ms against 0.3 ms.
constexpr int kFrWarps = 8;
constexpr int kFrChunk = 256;

struct ForceScreen {
  float fs[3];    // L / 2^32
  float screen2;  // r_c^2 + 0.01
};

__global__ void __launch_bounds__(kFrWarps * 32)
k_force_real(const double* __restrict__ xyz, const double* __restrict__ alpha,
             const uint32_t* __restrict__ sfix, int n, const double* __restrict__ ion_xyz,
             const uint32_t* __restrict__ sion, int n_ion, const double* __restrict__ q,
             double lx, double ly, double lz, double g, double rc, const ForceScreen fs,
             int nsplit, int per_warp, double* __restrict__ part, double2* __restrict__ slab,
             bool beside) {
  __shared__ uint4 su[kFrChunk];  // fixed-point x, y, z of the staged atoms
  __shared__ double sion_xyz[32][3];
  __shared__ int qa[kFrWarps][64];       // queued pairs: atom,
  __shared__ uint8_t ql[kFrWarps][64];   //   lane of the ion
  __shared__ double qv[kFrWarps][32][3];
  __shared__ double red[kFrWarps][32][3];
  wait_previous(beside);
  sion = fresh(sion);
  const int f = blockIdx.y, frames = gridDim.y, sp = blockIdx.z;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int I = blockIdx.x * 32 + lane;
  const bool live = I < n_ion;
  const size_t e = (size_t)f * n_ion + (live ? I : n_ion - 1);
  const uint32_t u0 = sion[3 * e], u1 = sion[3 * e + 1], u2 = sion[3 * e + 2];
  if (warp == 0)
    for (int d = 0; d < 3; ++d) sion_xyz[lane][d] = ion_xyz[3 * e + d];
  const double* qf = q + (size_t)f * n;
  const double L[3] = {lx, ly, lz};
  const double invL[3] = {1.0 / lx, 1.0 / ly, 1.0 / lz};
  const double rc2 = rc * rc;
  double gr[3] = {0.0, 0.0, 0.0};
  auto drain = [&](int cnt) {
    __syncwarp();
    if (lane < cnt) {
      const int a = qa[warp][lane];
      const double* ri = sion_xyz[ql[warp][lane]];
      const double al = alpha[a], qa_ = qf[a];
      double d0[3], s[3] = {0.0, 0.0, 0.0};
      int lo[3], hi[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        d0[d] = xyz[3 * a + d] - ri[d];
        d0[d] -= L[d] * rint(d0[d] * invL[d]);
        lo[d] = (int)ceil((-rc - d0[d]) * invL[d]);
        hi[d] = (int)floor((rc - d0[d]) * invL[d]);
      }
      for (int ix = lo[0]; ix <= hi[0]; ++ix)
        for (int iy = lo[1]; iy <= hi[1]; ++iy)
          for (int iz = lo[2]; iz <= hi[2]; ++iz) {
            const double dx = d0[0] + ix * L[0], dy = d0[1] + iy * L[1], dz = d0[2] + iz * L[2];
            const double r2 = dx * dx + dy * dy + dz * dz;
            if (r2 >= rc2 || r2 == 0.0) continue;
            const double r = sqrt(r2);
            const double w = qa_ * radial_derivative(g, al, r) / r;
            s[0] -= w * dx;
            s[1] -= w * dy;
            s[2] -= w * dz;
          }
#pragma unroll
      for (int d = 0; d < 3; ++d) qv[warp][lane][d] = s[d];
    }
    __syncwarp();
    for (int k = 0; k < cnt; ++k)
      if (ql[warp][k] == lane)
#pragma unroll
        for (int d = 0; d < 3; ++d) gr[d] += qv[warp][k][d];
    __syncwarp();
  };
  const int a0 = (int)((int64_t)n * sp / nsplit), a1 = (int)((int64_t)n * (sp + 1) / nsplit);
  int qn = 0;
  double qz = 0.0, qs = 0.0;  // this thread's share of sum q_i z_i and sum q_i
  const int chunk = kFrWarps * per_warp;
  for (int base = a0; base < a1; base += chunk) {
    const int i = base + (int)threadIdx.x;
    __syncthreads();
    if (i < a1 && (int)threadIdx.x < chunk) {
      su[threadIdx.x] = make_uint4(sfix[3 * i], sfix[3 * i + 1], sfix[3 * i + 2], 0u);
      if (blockIdx.x == 0) {
        qz += qf[i] * xyz[3 * i + 2];
        qs += qf[i];
      }
    }
    __syncthreads();
    const int t1 = min(per_warp, a1 - base - warp * per_warp);
    for (int t = 0; t < t1; ++t) {
      const uint4 ua = su[warp * per_warp + t];
      const float dx = (float)(int32_t)(ua.x - u0) * fs.fs[0];
      const float dy = (float)(int32_t)(ua.y - u1) * fs.fs[1];
      const float dz = (float)(int32_t)(ua.z - u2) * fs.fs[2];
      const bool in = live && fmaf(dz, dz, fmaf(dy, dy, dx * dx)) < fs.screen2;
      const unsigned m = __ballot_sync(0xffffffffu, in);
      if (!m) continue;
      if (in) {
        const int at = qn + __popc(m & ((1u << lane) - 1u));
        qa[warp][at] = base + warp * per_warp + t;
        ql[warp][at] = (uint8_t)lane;
      }
      qn += __popc(m);
      if (qn >= 32) {
        drain(32);
        if (lane < qn - 32) {
          qa[warp][lane] = qa[warp][32 + lane];
          ql[warp][lane] = ql[warp][32 + lane];
        }
        qn -= 32;
        __syncwarp();
      }
    }
  }
  if (qn > 0) drain(qn);
#pragma unroll
  for (int d = 0; d < 3; ++d) red[warp][lane][d] = gr[d];
  __syncthreads();
  if (threadIdx.x < 96 && blockIdx.x * 32 + (int)threadIdx.x / 3 < n_ion) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kFrWarps; ++w) s += red[w][threadIdx.x / 3][threadIdx.x % 3];
    part[(((size_t)sp * frames + f) * n_ion + blockIdx.x * 32) * 3 + threadIdx.x] = s;
  }
  if (blockIdx.x == 0) {  // the share's slab sums, warps in order
    for (int o = 16; o; o >>= 1) {
      qz += __shfl_xor_sync(0xffffffffu, qz, o);
      qs += __shfl_xor_sync(0xffffffffu, qs, o);
    }
    __syncthreads();
    if (lane == 0) {
      red[warp][0][0] = qz;
      red[warp][0][1] = qs;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double2 s = make_double2(0.0, 0.0);
      for (int w = 0; w < kFrWarps; ++w) {
        s.x += red[w][0][0];
        s.y += red[w][0][1];
      }
      slab[(size_t)sp * frames + f] = s;
    }
  }
}

// F_I = -q_I grad_I from the shares of both parts, in share order, and the slab term of
// Eq. 39: grad_z += (4 pi / V) (sum_i q_i z_i - z_I sum_i q_i).
__global__ void k_force_finish(const double* __restrict__ ion_xyz,
                               const double* __restrict__ ion_q, int frames, int n_ion,
                               const double* __restrict__ kpart, int nk,
                               const double* __restrict__ rpart, const double2* __restrict__ slab,
                               int nr, double3 kscale, double slab_factor,
                               double* __restrict__ out) {
  wait_previous(false);
  kpart = fresh(kpart);
  rpart = fresh(rpart);
  slab = fresh(slab);
  const int64_t count = (int64_t)frames * n_ion;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < 3 * count;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t ion = e / 3;
    const int d = (int)(e % 3);
    double gk = 0.0, gr = 0.0;
    for (int s = 0; s < nk; ++s) gk += kpart[s * 3 * count + e];
    for (int s = 0; s < nr; ++s) gr += rpart[s * 3 * count + e];
    double g = gr + gk * (d == 0 ? kscale.x : d == 1 ? kscale.y : kscale.z);
    if (d == 2 && slab_factor != 0.0) {
      const int f = (int)(ion / n_ion);
      double2 t = make_double2(0.0, 0.0);
      for (int s = 0; s < nr; ++s) {
        const double2 p = slab[(size_t)s * frames + f];
        t.x += p.x;
        t.y += p.y;
      }
      g += slab_factor * (t.x - t.y * ion_xyz[e]);
    }
    out[e] = -ion_q[ion] * g;
  }
}

}  // namespace

// Shares of the long sums: enough blocks for eight waves of `sms` SMs where the ions alone
// do not give them (k-space: at least 1,024 k-vectors a share, so that a block's reduction
// of its 24 sums stays small beside them; real space: at least 32 atoms, four a warp).
ForceSplits force_splits(bool fp64, int n, int frames, int n_ion, int mpad, int kh, int sms) {
  ForceSplits s;
  const int64_t want = 8 * (int64_t)sms;
  const int64_t kblocks = (int64_t)frames * (fp64 ? n_ion : (n_ion + kFkIons - 1) / kFkIons);
  s.k_tail = (int)std::max<int64_t>(1, std::min<int64_t>((want + kblocks - 1) / kblocks,
                                                         std::max(1, (mpad - kh) / 1024)));
  s.k_total = s.k_tail + (!fp64 && kh > 0 ? 1 : 0);
  const int64_t rblocks = (int64_t)frames * ((n_ion + 31) / 32);
  s.real = (int)std::max<int64_t>(1, std::min<int64_t>((want + rblocks - 1) / rblocks,
                                                       (n + 31) / 32));
  // a share in whole chunks where it has several, else as evenly as its warps can
  const int share = (n + s.real - 1) / s.real;
  s.real_per_warp = std::max(4, std::min(32, (share + kFrWarps - 1) / kFrWarps));
  return s;
}

// Launched after the ions' fixed-point coordinates, which it waits for; beside: what comes after
// may start beside it.
void launch_force_real(const double* xyz, const double* alpha, const uint32_t* sfix, int n,
                       const double* ion_xyz, const uint32_t* sion, int frames, int n_ion,
                       const double* q, const Geometry& geo, const ForceSplits& sp, double* rpart,
                       double2* slab, bool beside, cudaStream_t s) {
  ForceScreen fs;
  for (int d = 0; d < 3; ++d) fs.fs[d] = (float)(geo.L[d] * 0x1p-32);
  fs.screen2 = (float)(geo.rc * geo.rc) + 0.01f;
  launch_next(k_force_real, dim3((n_ion + 31) / 32, frames, sp.real), kFrWarps * 32, 0, s, xyz, alpha,
              sfix, n, ion_xyz, sion, n_ion, q, geo.L[0], geo.L[1], geo.L[2], geo.g, geo.rc, fs,
              sp.real, sp.real_per_warp, rpart, slab, beside);
}

void launch_force_kspace_and_finish(bool fp64, const double* ion_xyz, const double* ion_q,
                                    const uint32_t* sion, int frames, int n_ion, const int* hkl,
                                    const double* sqw, int mpad, int kh, const Geometry& geo,
                                    const void* turn, const void* v, const void* vhead,
                                    const double2* ion_axis, const AxisPhasors& ap,
                                    const ForceSplits& sp, double* kpart, const double* rpart,
                                    const double2* slab, double* out, cudaStream_t s) {
  if (fp64)
    launch_next(k_force_kspace_f64, dim3(n_ion, frames, sp.k_tail), kFkThreads, 0, s, ion_axis, ap,
                n_ion, hkl, sqw, mpad, sp.k_tail, (const double*)v, kpart);
  else
    launch_next(k_force_kspace, dim3((n_ion + kFkIons - 1) / kFkIons, frames, sp.k_total), kFkThreads,
                0, s, sion, n_ion, hkl, sqw, mpad, kh, sp.k_tail, (const float4*)turn,
                (const float*)v, (const float2*)vhead, kpart);
  const double twopi = 2.0 * kPi;
  const int64_t len = 3 * (int64_t)frames * n_ion;
  launch_next(k_force_finish, dim3((int)std::min<int64_t>((len + 127) / 128, 8192)), 128, 0, s,
              ion_xyz, ion_q, frames, n_ion, (const double*)kpart, sp.k_total, rpart, slab, sp.real,
              make_double3(twopi / geo.L[0], twopi / geo.L[1], twopi / geo.L[2]),
              geo.slab ? 4.0 * kPi / (geo.L[0] * geo.L[1] * geo.L[2]) : 0.0, out);
}

}  // namespace cpm
