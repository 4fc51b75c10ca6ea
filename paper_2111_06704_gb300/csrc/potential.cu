// Electrolyte potential on the electrode atoms (Eq. 25):
//   b^sol_i = sum_I q_I e_iI(alpha_i),   b_i = chi_i - k_e b^sol_i,
// with e_iI the point-Gaussian Ewald coefficient (alpha_iI = alpha_i) in the
// neutral-equivalent form (slab: dipole term (4 pi/V) z_i z_I only).
//
// Reciprocal part: ion structure factors v = [sqrt(W) Re S | sqrt(W) Im S],
// S_K = sum_I q_I exp(i K.r_I), then b^sol_k = A v with the electrode operand A of the
// E build (cos(K.(r_i - r_I)) split by angle addition).  Real part: direct pair sums
// over the images within the cutoff.
#include <math.h>

#include <algorithm>

#include "phasor.cuh"

namespace cpm {

namespace {

constexpr int kSfThreads = 128;
constexpr int kIonChunk = 256;

// Fractional ion coordinates in 2^-32 fixed point, once per ion and frame: the phases of
// every k-vector and the real-space screening use them.
__global__ void k_ion_fixed(const double* __restrict__ ion_xyz, int64_t count, double lx,
                            double ly, double lz, uint32_t* __restrict__ sion) {
  const double L[3] = {lx, ly, lz};
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < 3 * count;
       e += (int64_t)gridDim.x * blockDim.x) {
    double s = ion_xyz[e] / L[e % 3];
    s -= floor(s);
    sion[e] = (uint32_t)((unsigned long long)llrint(s * 4294967296.0) & 0xffffffffull);
  }
}

// exp(2 pi i j / 4096), j < 4096, as float pairs (cos hi, cos lo, sin hi, sin lo).
__global__ void k_turn_table(float4* __restrict__ T) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= 4096) return;
  double s, c;
  sincospi(j / 2048.0, &s, &c);
  const float ch = (float)c, sh = (float)s;
  T[j] = make_float4(ch, (float)(c - ch), sh, (float)(s - sh));
}

constexpr int kSfBlock = 8;  // ions a float block sum of the tail k-vectors holds

// sin and cos of 2 pi ph 2^-32 from a 64-entry table of exp(2 pi i j / 64) (float cos and
// sin, in shared memory: 512 bytes, few bank conflicts for random entries) and the
// remaining angle t = 2 pi (ph mod 2^26) 2^-32 < 0.099 rad by angle addition, with
// cos t = 1 - t^2/2 + t^4/24 and sin t = t - t^3/6 + t^5/120 (the next terms, t^6/720 and
// t^7/5040, lie below float rounding).  At most 1.5 float ulp of 1 (0.5 on average).
__device__ __forceinline__ void sincos_t64(uint32_t ph, const float2* T, float* s, float* c) {
  const float2 e = T[ph >> 26];
  const float t = (float)(ph & 0x3FFFFFFu) * 1.462918119976564e-09f;  // 2 pi 2^-32
  const float t2 = t * t;
  const float ct = fmaf(t2, fmaf(t2, 1.0f / 24.0f, -0.5f), 1.0f);
  const float st = t * fmaf(t2, fmaf(t2, 1.0f / 120.0f, -1.0f / 6.0f), 1.0f);
  *c = fmaf(e.x, ct, -(e.y * st));
  *s = fmaf(e.y, ct, e.x * st);
}

// v[f][c(k)] = sqrt(W_k) sum_I q_I cos(theta_Ik), v[f][c(k) + 64] = sqrt(W_k) sum_I q_I sin,
// in the column layout of the electrode operand, c(k) = 128 (k / 64) + k % 64, from the
// exact fixed-point phases.  Sums over the ions run in error-free float pairs (S_K is a
// sum of O(n_ion) unit phasors whose float partial sums would lose bits; FP64 runs at
// 1/64 of the float rate here); the tail's terms go in float blocks of kSfBlock ions, each
// block's sum into the pair (a few ulp of a block, not of the whole sum).  The tail
// k-vectors take float sin/cos from the phasor table (sincos_table, about one ulp); the
// head (k < kh, the heaviest weights) takes float-pair phasors and goes out in FP64 to
// vhead for the FP64 head contraction.
__global__ void __launch_bounds__(kSfThreads, 8)
k_ion_sf_f32(const uint32_t* __restrict__ sion, int64_t coord_stride,
             const double* __restrict__ ion_q, int n_ion,
             const int* __restrict__ hkl, const double* __restrict__ sqw, int mpad, int kh,
             const float4* __restrict__ turn, float* __restrict__ vout,
             double* __restrict__ vhead) {
  __shared__ uint32_t sf[kIonChunk][3];
  __shared__ float sqh[kIonChunk], sql[kIonChunk];
  __shared__ float2 t64[64];  // exp(2 pi i j / 64): entries 64 j of the 4,096-entry table
  const int f = blockIdx.y;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t* fx = sion + (size_t)f * coord_stride * 3;
  const double* q = ion_q + (size_t)f * n_ion;
  for (int j = threadIdx.x; j < 64; j += blockDim.x) {
    const float4 e = __ldg(turn + 64 * j);
    t64[j] = make_float2(e.x, e.z);
  }
  uint32_t h = 0, kk = 0, l = 0;
  if (k < mpad) {
    h = (uint32_t)hkl[3 * k];
    kk = (uint32_t)hkl[3 * k + 1];
    l = (uint32_t)hkl[3 * k + 2];
  }
  const bool head = k < kh;  // whole blocks take one branch unless they straddle kh
  float reh = 0.f, rel = 0.f, imh = 0.f, iml = 0.f;
  float rlo = 0.f, ilo = 0.f;  // tail: the charges' low parts times the phasors
  for (int base = 0; base < n_ion; base += kIonChunk) {
    const int cnt = min(kIonChunk, n_ion - base);
    __syncthreads();
    for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
      sf[t][0] = fx[3 * (base + t)];
      sf[t][1] = fx[3 * (base + t) + 1];
      sf[t][2] = fx[3 * (base + t) + 2];
      const double qv = q[base + t];
      sqh[t] = (float)qv;
      sql[t] = (float)(qv - (double)sqh[t]);
    }
    __syncthreads();
    if (k >= mpad) continue;
    if (head) {
      for (int t = 0; t < cnt; ++t) {
        const uint32_t ph = h * sf[t][0] + kk * sf[t][1] + l * sf[t][2];
        float ch, cl, sh, sl, ph_, pl_;
        phasor_ff(ph, turn, ch, cl, sh, sl);
        ff_mul(sqh[t], sql[t], ch, cl, ph_, pl_);
        ff_add(reh, rel, ph_, pl_, reh, rel);
        ff_mul(sqh[t], sql[t], sh, sl, ph_, pl_);
        ff_add(imh, iml, ph_, pl_, imh, iml);
      }
    } else {
      // blocks of kSfBlock ions summed in float, then added to the pairs by a two-sum;
      // the charges' low parts (zero for charges that are floats) summed in float apart
      int t = 0;
      for (; t + kSfBlock <= cnt; t += kSfBlock) {
        float br = 0.f, bi = 0.f;
#pragma unroll
        for (int u = 0; u < kSfBlock; ++u) {
          const uint32_t ph = h * sf[t + u][0] + kk * sf[t + u][1] + l * sf[t + u][2];
          float sn, cs;
          sincos_t64(ph, t64, &sn, &cs);
          br = fmaf(sqh[t + u], cs, br);
          bi = fmaf(sqh[t + u], sn, bi);
          rlo = fmaf(sql[t + u], cs, rlo);
          ilo = fmaf(sql[t + u], sn, ilo);
        }
        pair_add1(reh, rel, br);
        pair_add1(imh, iml, bi);
      }
      for (; t < cnt; ++t) {
        const uint32_t ph = h * sf[t][0] + kk * sf[t][1] + l * sf[t][2];
        float sn, cs;
        sincos_t64(ph, t64, &sn, &cs);
        pair_fma(reh, rel, sqh[t], sql[t], cs);
        pair_fma(imh, iml, sqh[t], sql[t], sn);
      }
    }
  }
  if (k >= mpad) return;
  const double re = (double)reh + (double)rel + (double)rlo,
               im = (double)imh + (double)iml + (double)ilo;
  const double w = sqw[k];
  const size_t kcol = 128 * (size_t)(k >> 6) + (k & 63);  // operand column layout
  float* v = vout + (size_t)f * 2 * mpad;
  if (head) {  // FP64 values for the FP64 head contraction; zero float columns
    double* vh = vhead + (size_t)f * 2 * kh;
    vh[kcol] = w * re;
    vh[kcol + 64] = w * im;
    v[kcol] = 0.f;
    v[kcol + 64] = 0.f;
  } else {
    v[kcol] = (float)(w * re);
    v[kcol + 64] = (float)(w * im);
  }
}

// exp(2 pi i j s_d) of every point and axis entry, s_d the fractional coordinate (from the
// positions, or from fixed-point coordinates where sfix is given): one sincospi per entry, a
// few hundred a point, instead of one per k-vector.
__global__ void k_axis_phasors(const double* __restrict__ xyz, const uint32_t* __restrict__ sfix,
                               int64_t count, double lx, double ly, double lz,
                               const AxisPhasors ap, double2* __restrict__ out) {
  const int64_t len = count * ap.len;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < len;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t pt = e / ap.len;
    const int j = (int)(e - pt * ap.len);
    const int d = j >= ap.off[2] ? 2 : j >= ap.off[1] ? 1 : 0;
    double s;
    if (sfix) {
      s = sfix[3 * pt + d] * 0x1p-32;
    } else {
      s = xyz[3 * pt + d] / (d == 0 ? lx : d == 1 ? ly : lz);
      s -= floor(s);
    }
    double fr = (j - ap.off[d]) * s;
    fr -= rint(fr);
    double sn, cs;
    sincospi(2.0 * fr, &sn, &cs);
    out[e] = make_double2(cs, sn);
  }
}

// FP64 storage (the plain baseline build): the same sums in FP64, the phasors as products of
// the points' per-axis phasors.  32 k-vectors a block (one a lane), the points dealt to its
// eight warps, whose sums are added in warp order: with one thread a k-vector over all
// points a 512-atom cell kept half of the chip busy.
constexpr int kSf64Warps = 8;

__global__ void __launch_bounds__(kSf64Warps * 32)
k_ion_sf_f64(const double2* __restrict__ axis, const AxisPhasors ap, int64_t coord_stride,
             const double* __restrict__ ion_q, int n_ion, const int* __restrict__ hkl,
             const double* __restrict__ sqw, int mpad, double* __restrict__ vout) {
  __shared__ double2 red[kSf64Warps][32];
  const int f = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k = blockIdx.x * 32 + lane;  // mpad is a multiple of 64
  const double2* tab = axis + (size_t)f * coord_stride * ap.len;
  const double* q = ion_q + (size_t)f * n_ion;
  const int h0 = hkl[3 * k], h1 = hkl[3 * k + 1], h2 = hkl[3 * k + 2];
  double re = 0.0, im = 0.0;
  for (int t = warp; t < n_ion; t += kSf64Warps) {
    const double2 e = ap.phasor(tab + (size_t)t * ap.len, h0, h1, h2);
    const double qt = q[t];
    re += qt * e.x;
    im += qt * e.y;
  }
  red[warp][lane] = make_double2(re, im);
  __syncthreads();
  if (warp != 0) return;
  for (int w = 1; w < kSf64Warps; ++w) {
    re += red[w][lane].x;
    im += red[w][lane].y;
  }
  const double w = sqw[k];
  const size_t kcol = 128 * (size_t)(k >> 6) + (k & 63);
  double* v = vout + (size_t)f * 2 * mpad;
  v[kcol] = w * re;
  v[kcol + 64] = w * im;
}

// b^sol_k[f][i] = sum_c A[i][c] v[f][c]: one warp per electrode row and NF frames per
// grid row (the A row is read once per NF frames).  Float storage: 4-term float partials
// summed in error-free float pairs; FP64 storage: FP64 throughout.
template <typename T, int NF>
__global__ void __launch_bounds__(256)
k_bsol_kspace(const T* __restrict__ A, int n, int64_t lda, const T* __restrict__ v,
              int frames, double* __restrict__ bsol, int accumulate) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int f0 = blockIdx.y * NF;
  if (warp >= n) return;
  const T* a = A + (int64_t)warp * lda;
  constexpr int VEC = 16 / sizeof(T);
  T hi[NF], lo[NF];
#pragma unroll
  for (int r = 0; r < NF; ++r) hi[r] = lo[r] = T(0);
  for (int64_t c = lane * VEC; c < lda; c += 32 * VEC) {
    T av[VEC];
    *reinterpret_cast<float4*>(av) = __ldg(reinterpret_cast<const float4*>(a + c));
#pragma unroll
    for (int r = 0; r < NF; ++r) {
      if (f0 + r >= frames) break;
      T vv[VEC];
      *reinterpret_cast<float4*>(vv) =
          __ldg(reinterpret_cast<const float4*>(v + (int64_t)(f0 + r) * lda + c));
      T s = T(0);
#pragma unroll
      for (int u = 0; u < VEC; ++u) s = fma(av[u], vv[u], s);
      if constexpr (sizeof(T) == 4) {
        const float t = hi[r] + s;
        const float bb = t - hi[r];
        lo[r] += (hi[r] - (t - bb)) + (s - bb);
        hi[r] = t;
      } else {
        hi[r] += s;
      }
    }
  }
#pragma unroll
  for (int r = 0; r < NF; ++r) {
    double x = (double)hi[r] + (double)lo[r];
    for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (lane == 0 && f0 + r < frames) {
      double* dst = bsol + (int64_t)(f0 + r) * n + warp;
      *dst = accumulate ? *dst + x : x;
    }
  }
}

// Streamed builds keep no A: b^sol_k[f][i] = sum_{k >= kh} sqrt(W_k) [cos(K.r_i) v_c +
// sin(K.r_i) v_s] with the electrode phases formed on the fly (fixed point, sincos_table);
// the terms of kDirectBlock consecutive k-vectors are summed in float, and each block's
// sum goes into an error-free float pair (a two-sum), so the rounding of the plain sums
// grows with the block, not with the ~10^5 k-vectors.  One thread per electrode atom and up to
// kDirectFrames frames per block: each phasor is formed once and used for every frame of
// the block; the k-vectors of a chunk and their structure factors are staged in shared
// memory.  Frames go in pairs through paired float instructions (two IEEE results an
// instruction, a - b as fma(b, -1, a)): the values are those of one frame at a time.
constexpr int kDirectChunk = 128;
constexpr int kDirectFrames = 16;
constexpr int kDirectBlock = 8;  // divides every chunk: head and table ends are multiples of 16

__global__ void __launch_bounds__(128, 4)
k_bsol_kspace_direct(const uint32_t* __restrict__ sfix, int n, const int* __restrict__ hkl,
                     const double* __restrict__ sqw, int mpad, int kh,
                     const float4* __restrict__ turn, const float* __restrict__ v, int frames,
                     double* __restrict__ bsol, int nsplit, int64_t split_stride) {
  __shared__ uint32_t sh[kDirectChunk][3];
  // sqrt(W) (v_cos, v_sin) of frames 2 p and 2 p + 1: (c_2p, c_2p+1, s_2p, s_2p+1)
  __shared__ float4 sv[kDirectChunk][kDirectFrames / 2];
  const int f0 = blockIdx.y * kDirectFrames;
  const int nf = min(kDirectFrames, frames - f0);
  // block = atom block + nblk x share: share sp takes chunks [c0, c1) of the k range
  const int nblk = gridDim.x / nsplit, sp = blockIdx.x / nblk;
  const int i = (blockIdx.x - sp * nblk) * blockDim.x + threadIdx.x;
  const int nch = (mpad - kh + kDirectChunk - 1) / kDirectChunk;
  const int kbeg = kh + (int)((int64_t)sp * nch / nsplit) * kDirectChunk;
  const int kend = min(mpad, kh + (int)((int64_t)(sp + 1) * nch / nsplit) * kDirectChunk);
  double* out = bsol + sp * split_stride;
  uint32_t u0 = 0, u1 = 0, u2 = 0;
  if (i < n) {
    u0 = sfix[3 * i];
    u1 = sfix[3 * i + 1];
    u2 = sfix[3 * i + 2];
  }
  float2 hi[kDirectFrames / 2], lo[kDirectFrames / 2];
#pragma unroll
  for (int f = 0; f < kDirectFrames / 2; ++f) hi[f] = lo[f] = make_float2(0.f, 0.f);
  const float2 m1 = make_float2(-1.f, -1.f);
  for (int k0 = kbeg; k0 < kend; k0 += kDirectChunk) {
    const int cnt = min(kDirectChunk, kend - k0);
    __syncthreads();
    for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
      const int k = k0 + t;
      sh[t][0] = (uint32_t)hkl[3 * k];
      sh[t][1] = (uint32_t)hkl[3 * k + 1];
      sh[t][2] = (uint32_t)hkl[3 * k + 2];
    }
    for (int e = threadIdx.x; e < cnt * (kDirectFrames / 2); e += blockDim.x) {
      const int t = e / (kDirectFrames / 2), fp = e % (kDirectFrames / 2);
      const int k = k0 + t;
      const size_t kcol = 128 * (size_t)(k >> 6) + (k & 63);
      const float w = (float)sqw[k];
      float4 val = make_float4(0.f, 0.f, 0.f, 0.f);
      if (2 * fp < nf) {
        const float* vf = v + (size_t)(f0 + 2 * fp) * 2 * mpad;
        val.x = w * vf[kcol];
        val.z = w * vf[kcol + 64];
      }
      if (2 * fp + 1 < nf) {
        const float* vf = v + (size_t)(f0 + 2 * fp + 1) * 2 * mpad;
        val.y = w * vf[kcol];
        val.w = w * vf[kcol + 64];
      }
      sv[t][fp] = val;
    }
    __syncthreads();
    if (i >= n) continue;
    for (int tb = 0; tb < cnt; tb += kDirectBlock) {
      float2 blk[kDirectFrames / 2];
#pragma unroll
      for (int f = 0; f < kDirectFrames / 2; ++f) blk[f] = make_float2(0.f, 0.f);
#pragma unroll 2
      for (int tt = 0; tt < kDirectBlock; ++tt) {
        const int t = tb + tt;
        float sn, cs;
        sincos_table(sh[t][0] * u0 + sh[t][1] * u1 + sh[t][2] * u2, turn, &sn, &cs);
        const float2 sn2 = make_float2(sn, sn), cs2 = make_float2(cs, cs);
#pragma unroll
        for (int f = 0; f < kDirectFrames / 2; ++f) {
          const float4 vv = sv[t][f];
          blk[f] = __ffma2_rn(sn2, make_float2(vv.z, vv.w),
                              __ffma2_rn(cs2, make_float2(vv.x, vv.y), blk[f]));
        }
      }
#pragma unroll
      for (int f = 0; f < kDirectFrames / 2; ++f) {
        const float2 term = blk[f];
        const float2 s2 = __fadd2_rn(hi[f], term);
        const float2 bb = __ffma2_rn(hi[f], m1, s2);                          // s2 - hi
        const float2 a = __ffma2_rn(__ffma2_rn(bb, m1, s2), m1, hi[f]);       // hi - (s2 - bb)
        lo[f] = __fadd2_rn(lo[f], __fadd2_rn(a, __ffma2_rn(bb, m1, term)));   // + (term - bb)
        hi[f] = s2;
      }
    }
  }
  if (i < n)
#pragma unroll
    for (int f = 0; f < kDirectFrames; ++f) {
      const float h = (f & 1) ? hi[f >> 1].y : hi[f >> 1].x;
      const float l = (f & 1) ? lo[f >> 1].y : lo[f >> 1].x;
      if (f < nf) out[(size_t)(f0 + f) * n + i] = (double)h + (double)l;
    }
}

}  // namespace

void launch_ion_fixed(const double* ion_xyz, int frames, int n_ion, const double L[3],
                      uint32_t* sion, cudaStream_t s) {
  const int64_t count = (int64_t)frames * n_ion;
  const int blocks = (int)std::min<int64_t>((3 * count + 255) / 256, 4096);
  (k_ion_fixed<<<blocks, 256, 0, s>>>(ion_xyz, count, L[0], L[1], L[2], sion), note_launch());
}

void launch_turn_table(void* T, cudaStream_t s) {
  (k_turn_table<<<16, 256, 0, s>>>((float4*)T), note_launch());
}

void launch_axis_phasors(const double* xyz, const uint32_t* sfix, int64_t count,
                         const double L[3], const AxisPhasors& ap, double2* out,
                         cudaStream_t s) {
  const int blocks = (int)std::min<int64_t>((count * ap.len + 127) / 128, 16384);
  (k_axis_phasors<<<blocks, 128, 0, s>>>(xyz, sfix, count, L[0], L[1], L[2], ap, out), note_launch());
}

void launch_ion_structure_factor(bool fp64, const double2* axis, const AxisPhasors& ap,
                                 const uint32_t* sion, int64_t coord_stride,
                                 const double* ion_q, int frames, int n_ion, const int* hkl,
                                 const double* sqw, int mpad, int kh, const void* turn,
                                 void* v, double* vhead, cudaStream_t s) {
  if (fp64) {
    (k_ion_sf_f64<<<dim3(mpad / 32, frames), kSf64Warps * 32, 0, s>>>(
         axis, ap, coord_stride, ion_q, n_ion, hkl, sqw, mpad, (double*)v),
     note_launch());
  } else {
    dim3 grid((mpad + kSfThreads - 1) / kSfThreads, frames);
    (k_ion_sf_f32<<<grid, kSfThreads, 0, s>>>(sion, coord_stride, ion_q, n_ion, hkl, sqw, mpad,
                                              kh, (const float4*)turn, (float*)v, vhead),
     note_launch());
  }
}

namespace {

// The k-range shares of the direct sum, summed in share order into b^sol_k.
__global__ void k_sum_splits(const double* __restrict__ part, int nsplit, int64_t stride,
                             int64_t count, double* __restrict__ out) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count;
       e += (int64_t)gridDim.x * blockDim.x) {
    double v = part[e];
    for (int sp = 1; sp < nsplit; ++sp) v += part[sp * stride + e];
    out[e] = v;
  }
}

}  // namespace

// Shares of the k range for the direct sum: the atom blocks of kDirectFrames-frame groups
// (four resident an SM) times the shares fill whole waves of `sms` SMs best (a larger
// count only where it fills 2% more of the last wave).
int bsol_direct_splits(int n, int frames, int mpad, int kh, int sms) {
  const int64_t blocks = (int64_t)((n + 127) / 128) * ((frames + kDirectFrames - 1) / kDirectFrames);
  const int nch = (mpad - kh + kDirectChunk - 1) / kDirectChunk;
  const int64_t cap = 4 * (int64_t)sms;
  int best = 1;
  double best_eff = -1.0;
  for (int sp = 1; sp <= std::min(4, std::max(1, nch)); ++sp) {
    const int64_t units = blocks * sp, waves = (units + cap - 1) / cap;
    const double eff = (double)units / (double)(waves * cap);
    if (eff > best_eff + 0.02) {
      best_eff = eff;
      best = sp;
    }
  }
  return best;
}

// b^sol_k = A v: in float storage the head k-vectors (the heaviest weights) are
// contracted in FP64 against an FP64 copy of their operand columns.  Without A (a streamed
// build) the float part is the direct sum over the tail k-vectors.
void launch_bsol_kspace(bool fp64, const void* A, const double* Ahead, int n, int mpad, int kh,
                        const void* v, const double* vhead, int frames, double* bsol,
                        const uint32_t* sfix, const int* hkl, const double* sqw,
                        const void* turn, int nsplit, double* split_part, cudaStream_t s) {
  const int64_t lda = 2 * (int64_t)mpad;
  if (!A && !fp64) {
    const int fgroups = (frames + kDirectFrames - 1) / kDirectFrames;
    const int sp = split_part ? nsplit : 1;
    const int64_t stride = (int64_t)frames * n;  // between shares
    double* dst = sp > 1 ? split_part : bsol;
    for (int g0 = 0; g0 < fgroups; g0 += 65535) {
      const int f0 = g0 * kDirectFrames;
      (k_bsol_kspace_direct<<<dim3(sp * ((n + 127) / 128), std::min(fgroups - g0, 65535)), 128,
                              0, s>>>(sfix, n, hkl, sqw, mpad, kh, (const float4*)turn,
                                      (const float*)v + f0 * lda, frames - f0,
                                      dst + (int64_t)f0 * n, sp, stride),
       note_launch());
    }
    if (sp > 1)
      (k_sum_splits<<<(int)std::min<int64_t>((stride + 255) / 256, 8192), 256, 0, s>>>(
           split_part, sp, stride, stride, bsol),
       note_launch());
    for (int g0 = 0; kh > 0 && g0 < (frames + 3) / 4; g0 += 65535) {
      const int f0 = 4 * g0;
      const dim3 grid((n * 32 + 255) / 256, std::min((frames - f0 + 3) / 4, 65535));
      (k_bsol_kspace<double, 4><<<grid, 256, 0, s>>>(Ahead, n, 2 * (int64_t)kh,
                                                     vhead + f0 * 2 * (int64_t)kh, frames - f0,
                                                     bsol + (int64_t)f0 * n, 1), note_launch());
    }
    return;
  }
  for (int g0 = 0; g0 < (frames + 3) / 4; g0 += 65535) {
    const int f0 = 4 * g0;
    const dim3 grid((n * 32 + 255) / 256, std::min((frames - f0 + 3) / 4, 65535));
    if (fp64) {
      (k_bsol_kspace<double, 4><<<grid, 256, 0, s>>>((const double*)A, n, lda,
                                                     (const double*)v + f0 * lda, frames - f0,
                                                     bsol + (int64_t)f0 * n, 0), note_launch());
    } else {
      (k_bsol_kspace<float, 4><<<grid, 256, 0, s>>>((const float*)A, n, lda,
                                                    (const float*)v + f0 * lda, frames - f0,
                                                    bsol + (int64_t)f0 * n, 0), note_launch());
      if (kh > 0)
        (k_bsol_kspace<double, 4><<<grid, 256, 0, s>>>(Ahead, n, 2 * (int64_t)kh,
                                                       vhead + f0 * 2 * (int64_t)kh, frames - f0,
                                                       bsol + (int64_t)f0 * n, 1), note_launch());
    }
  }
}

}  // namespace cpm
