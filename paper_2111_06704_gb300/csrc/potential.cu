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
#include <type_traits>

#include "phasor.cuh"
#include "programmatic.cuh"

namespace cpm {

namespace {

// Fractional ion coordinates in 2^-32 fixed point, once per ion and frame: the phases of
// every k-vector and the real-space screening use them.
__global__ void k_ion_fixed(const double* __restrict__ ion_xyz, int64_t count, double lx,
                            double ly, double lz, uint32_t* __restrict__ sion) {
  set_up_next();
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

constexpr int kSfWarps = 8;
constexpr int kSfBlock = 8;   // ions a float block sum of the tail k-vectors holds
constexpr int kIonChunk = 256;

// sin and cos of 2 pi ph 2^-32 for two phases from a 64-entry table of exp(2 pi i j / 64) and
// the remaining angle t = 2 pi (ph mod 2^26) 2^-32 < 0.099 rad by angle addition, with
// cos t = 1 - t^2/2 + t^4/24 and sin t = t - t^3/6 + t^5/120 (the next terms, t^6/720 and
// t^7/5040, lie below float rounding), in paired instructions.  At most 1.5 float ulp of 1
// (0.5 on average).  tc and ts point at the lane's own copy of the table in shared memory
// (entry j at [32 j]), so no two lanes meet in a bank.
__device__ __forceinline__ void sincos_t64x2(uint32_t p0, uint32_t p1, const float* tc,
                                             const float* ts, float2& s, float2& c) {
  const int i0 = (int)(p0 >> 26) * 32, i1 = (int)(p1 >> 26) * 32;
  const float2 ex = make_float2(tc[i0], tc[i1]), ey = make_float2(ts[i0], ts[i1]);
  const float2 u = make_float2((float)(p0 & 0x3FFFFFFu), (float)(p1 & 0x3FFFFFFu));
  const float k = 1.462918119976564e-09f;  // 2 pi 2^-32
  const float2 t = __fmul2_rn(u, make_float2(k, k));
  const float2 t2 = __fmul2_rn(t, t);
  const float2 ct = __ffma2_rn(
      t2, __ffma2_rn(t2, make_float2(1.0f / 24.0f, 1.0f / 24.0f), make_float2(-0.5f, -0.5f)),
      make_float2(1.0f, 1.0f));
  const float2 st = __fmul2_rn(
      t, __ffma2_rn(t2,
                    __ffma2_rn(t2, make_float2(1.0f / 120.0f, 1.0f / 120.0f),
                               make_float2(-1.0f / 6.0f, -1.0f / 6.0f)),
                    make_float2(1.0f, 1.0f)));
  const float2 neg = make_float2(-ey.x, -ey.y);
  c = __ffma2_rn(ex, ct, __fmul2_rn(neg, st));
  s = __ffma2_rn(ey, ct, __fmul2_rn(ex, st));
}

// v[f][c(k)] = sqrt(W_k) sum_I q_I cos(theta_Ik), v[f][c(k) + 64] = sqrt(W_k) sum_I q_I sin,
// in the column layout of the electrode operand, c(k) = 128 (k / 64) + k % 64, from the
// exact fixed-point phases.  Sums over the ions run in error-free float pairs (S_K is a
// sum of O(n_ion) unit phasors whose float partial sums would lose bits; FP64 runs at
// 1/64 of the float rate here); the tail's terms go in float blocks of kSfBlock ions, each
// block's sum into the pair (a few ulp of a block, not of the whole sum).  The head (k < kh,
// the heaviest weights) takes float-pair phasors and goes out as float pairs to vhead for
// the head contraction.
//
// Bound by issue: 4.4e9 phasors a call at 512 atoms, 2,000 ions, 256 frames.  A thread takes
// two tail k-vectors with consecutive l (the list of pairs is the context's): one broadcast
// load of an ion, four integer operations for both phases instead of six multiply-adds, and
// paired float instructions throughout; the phasor table has a copy for every lane (random
// entries of one copy conflicted in the banks).  One k-vector a thread with a shared table
// took 3,995 us there, this form 3,473 (a phasor is 13 FMA-pipe operations, and a paired
// FMA of three registers takes 3 cycles; 217,619 k-vectors over 12,800 points 2,752 -> 2,261 us).  Where the k-vectors do not fill the chip, the warps
// of a block split the ions' blocks of eight between them (tail_shares).  The head's sums are chains of dependent additions (some 700
// cycles an ion among other warps: one thread a k-vector for all ions was 60% longer than
// the rest of the grid), so its blocks always split the ions eight ways, and come first.
__global__ void __launch_bounds__(kSfWarps * 32)
k_ion_sf_f32(const uint32_t* __restrict__ sion, int64_t coord_stride,
             const double* __restrict__ ion_q, int n_ion, const SfPair* __restrict__ pairs,
             int npairs, const int* __restrict__ hkl, const double* __restrict__ sqw, int mpad,
             int kh, int tail_shares, int head_blocks, const float4* __restrict__ turn,
             float* __restrict__ vout, float2* __restrict__ vhead, bool late,
             unsigned long long* stamp) {
  __shared__ uint4 si[kIonChunk];   // fixed-point x, y, z and the charge as a float
  __shared__ float sql[kIonChunk];  // the charges' low parts
  __shared__ float tc[64][32], ts[64][32];  // exp(2 pi i j / 64), a copy for every lane
  __shared__ double red[kSfWarps][32][4];
  if (!late) wait_previous(false);
  stamp_time(stamp);
  sion = fresh(sion);
  ion_q = fresh(ion_q);
  const int f = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool head = (int)blockIdx.x < head_blocks;
  const int shares = head ? kSfWarps : tail_shares;
  const int share = warp % shares, per = kSfWarps / shares;  // groups of 32 threads a block
  const uint32_t* fx = sion + (size_t)f * coord_stride * 3;
  const double* q = ion_q + (size_t)f * n_ion;
  float* v = vout + (size_t)f * 2 * mpad;
  const int at = ((int)blockIdx.x - (head ? 0 : head_blocks)) * per * 32 +
                 (warp / shares) * 32 + lane;
  uint32_t h = 0, kk = 0, l = 0;
  int k0 = -1, k1 = -1;
  if (head) {
    if (at < kh) {
      k0 = at;
      h = (uint32_t)hkl[3 * at];
      kk = (uint32_t)hkl[3 * at + 1];
      l = (uint32_t)hkl[3 * at + 2];
    }
  } else {
    for (int e = threadIdx.x; e < 64 * 32; e += kSfWarps * 32) {
      const float4 w = __ldg(turn + 64 * (e >> 5));
      tc[e >> 5][e & 31] = w.x;
      ts[e >> 5][e & 31] = w.z;
    }
    if (at < npairs) {
      const SfPair p = pairs[at];
      h = (uint32_t)p.h;
      kk = (uint32_t)p.k;
      l = (uint32_t)p.l;
      k0 = p.k0;
      k1 = p.k1;
    }
  }
  const float *tcl = &tc[0][lane], *tsl = &ts[0][lane];
  float2 reh = {0.f, 0.f}, rel = {0.f, 0.f}, imh = {0.f, 0.f}, iml = {0.f, 0.f};
  float2 rlo = {0.f, 0.f}, ilo = {0.f, 0.f};  // tail: the charges' low parts times the phasors
  for (int base = 0; base < n_ion; base += kIonChunk) {
    const int cnt = min(kIonChunk, n_ion - base);
    __syncthreads();
    int low = 0;
    for (int t = threadIdx.x; t < cnt; t += kSfWarps * 32) {
      const double qv = q[base + t];
      const float qh = (float)qv, qlo = (float)(qv - (double)qh);
      si[t] = make_uint4(fx[3 * (base + t)], fx[3 * (base + t) + 1], fx[3 * (base + t) + 2],
                         __float_as_uint(qh));
      sql[t] = qlo;
      low |= qlo != 0.f;
    }
    low = __syncthreads_or(low);  // any charge that is no float
    if (head) {
#pragma unroll 2
      for (int t = share; t < cnt; t += kSfWarps) {
        const uint4 e = si[t];
        const float qh = __uint_as_float(e.w), ql = sql[t];
        float ch, cl, sh, sl, ph, pl;
        phasor_ff(h * e.x + kk * e.y + l * e.z, turn, ch, cl, sh, sl);
        ff_mul(qh, ql, ch, cl, ph, pl);
        ff_add(reh.x, rel.x, ph, pl, reh.x, rel.x);
        ff_mul(qh, ql, sh, sl, ph, pl);
        ff_add(imh.x, iml.x, ph, pl, imh.x, iml.x);
      }
      continue;
    }
    const int blocks = cnt / kSfBlock;
    auto block = [&](int b, auto lowpart) {
      float2 br = make_float2(0.f, 0.f), bi = make_float2(0.f, 0.f);
#pragma unroll
      for (int u = 0; u < kSfBlock; ++u) {
        const uint4 e = si[b * kSfBlock + u];
        const uint32_t p0 = h * e.x + kk * e.y + l * e.z;
        float2 sn, cs;
        sincos_t64x2(p0, p0 + e.z, tcl, tsl, sn, cs);
        const float2 qq = make_float2(__uint_as_float(e.w), __uint_as_float(e.w));
        br = __ffma2_rn(qq, cs, br);
        bi = __ffma2_rn(qq, sn, bi);
        if constexpr (decltype(lowpart)::value) {
          const float ql = sql[b * kSfBlock + u];
          rlo = __ffma2_rn(make_float2(ql, ql), cs, rlo);
          ilo = __ffma2_rn(make_float2(ql, ql), sn, ilo);
        }
      }
      pair_add2(reh, rel, br);
      pair_add2(imh, iml, bi);
    };
    if (low)
      for (int b = share; b < blocks; b += shares) block(b, std::true_type());
    else
      for (int b = share; b < blocks; b += shares) block(b, std::false_type());
    if (share == blocks % shares)  // ions past the last whole block, each into the pair
      for (int t = blocks * kSfBlock; t < cnt; ++t) {
        const uint4 e = si[t];
        const uint32_t p0 = h * e.x + kk * e.y + l * e.z;
        float2 sn, cs;
        sincos_t64x2(p0, p0 + e.z, tcl, tsl, sn, cs);
        const float qh = __uint_as_float(e.w), ql = sql[t];
        pair_fma(reh.x, rel.x, qh, ql, cs.x);
        pair_fma(reh.y, rel.y, qh, ql, cs.y);
        pair_fma(imh.x, iml.x, qh, ql, sn.x);
        pair_fma(imh.y, iml.y, qh, ql, sn.y);
      }
  }
  double re[2] = {(double)reh.x + (double)rel.x + (double)rlo.x,
                  (double)reh.y + (double)rel.y + (double)rlo.y};
  double im[2] = {(double)imh.x + (double)iml.x + (double)ilo.x,
                  (double)imh.y + (double)iml.y + (double)ilo.y};
  if (shares > 1) {  // in share order
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      red[warp][lane][2 * u] = re[u];
      red[warp][lane][2 * u + 1] = im[u];
    }
    __syncthreads();
    if (share != 0) return;
    for (int s = 1; s < shares; ++s)
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        re[u] += red[warp + s][lane][2 * u];
        im[u] += red[warp + s][lane][2 * u + 1];
      }
  }
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int k = u == 0 ? k0 : k1;
    if (k < 0) continue;
    const double w = sqw[k];
    const size_t kcol = 128 * (size_t)(k >> 6) + (k & 63);  // operand column layout
    if (head) {  // float pairs for the head contraction; zero float columns
      float2* vh = vhead + (size_t)f * 2 * kh;
      const double c = w * re[u], sn = w * im[u];
      vh[kcol] = make_float2((float)c, (float)(c - (double)(float)c));
      vh[kcol + 64] = make_float2((float)sn, (float)(sn - (double)(float)sn));
      v[kcol] = 0.f;
      v[kcol + 64] = 0.f;
    } else {
      v[kcol] = (float)(w * re[u]);
      v[kcol + 64] = (float)(w * im[u]);
    }
  }
  end_after_previous(late);  // (warp 0 comes here: its share is the first)
}

// exp(2 pi i j s_d) of every point and axis entry, s_d the fractional coordinate (from the
// positions, or from fixed-point coordinates where sfix is given): one sincospi per entry, a
// few hundred a point, instead of one per k-vector.
__global__ void k_axis_phasors(const double* __restrict__ xyz, const uint32_t* __restrict__ sfix,
                               int64_t count, double lx, double ly, double lz,
                               const AxisPhasors ap, double2* __restrict__ out) {
  wait_previous(false);
  sfix = fresh(sfix);
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
// the points' per-axis phasors.  A lane takes an entry, the k-vectors (h, k, l) and (h, k, -l):
// with q exp(i (h x + k y)) = a + i b and exp(i l z) = c + i d the four sums of a c, b d, a d and
// b c over the points give both, two FP64 operations a k-vector and point.  a + i b is formed
// once a point and column (h, k) of the block's entries (32, sorted by column) and shared.
// The points are dealt to the block's eight warps, whose sums are added in warp order.  Bound by
// the FP64 pipe (two lanes a clock and SM): 84 us at 512 points, 8,645 k-vectors with ten
// operations a k-vector and point, 20 us so.
constexpr int kSf64Warps = 8;
constexpr int kSf64Batch = 8;  // points a warp takes at a time

__global__ void __launch_bounds__(kSf64Warps * 32)
k_ion_sf_f64(const double2* __restrict__ axis, const AxisPhasors ap, int64_t coord_stride,
             const double* __restrict__ ion_q, int64_t charge_stride, int n_ion, bool add,
             const SfEntry* __restrict__ entries,
             int nentries, const double* __restrict__ sqw, int m, int mpad,
             double* __restrict__ vout, bool late, unsigned long long* stamp) {
  __shared__ double2 s_ab[kSf64Warps][32][kSf64Batch];
  __shared__ double red[kSf64Warps][32][4];
  __shared__ int2 s_hk[32];  // the block's columns
  if (!late) wait_previous(false);
  stamp_time(stamp);
  axis = fresh(axis);
  vout = fresh(vout);
  const int f = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double* v = vout + (size_t)f * 2 * mpad;
  if (blockIdx.x == 0)  // the table's padding
    for (int k = m + (int)threadIdx.x; k < mpad; k += kSf64Warps * 32) {
      const size_t kcol = 128 * (size_t)(k >> 6) + (k & 63);
      v[kcol] = v[kcol + 64] = 0.0;
    }
  if (nentries == 0) return end_after_previous(late);
  const int e0 = blockIdx.x * 32;
  const SfEntry en = entries[min(e0 + lane, nentries - 1)];
  const int c0 = __shfl_sync(0xffffffffu, en.col, 0);
  const int ncol = __shfl_sync(0xffffffffu, en.col, 31) - c0 + 1, mine = en.col - c0;
  if (warp == 0) s_hk[mine] = make_int2(en.h, en.k);
  __syncthreads();
  const double2* tab = axis + (size_t)f * coord_stride * ap.len;
  const double* q = ion_q + (size_t)f * charge_stride;
  double ac = 0.0, bd = 0.0, ad = 0.0, bc = 0.0;
  for (int t0 = warp * kSf64Batch; t0 < n_ion; t0 += kSf64Warps * kSf64Batch) {
    const int cnt = min(kSf64Batch, n_ion - t0);
    __syncwarp();
    for (int e = lane; e < ncol * kSf64Batch; e += 32) {
      const int c = e / kSf64Batch, t = e % kSf64Batch;
      if (t >= cnt) continue;
      const double2* row = tab + (size_t)(t0 + t) * ap.len;
      const int2 hk = s_hk[c];
      double2 x = __ldca(row + ap.off[0] + abs(hk.x)), y = __ldca(row + ap.off[1] + abs(hk.y));
      if (hk.x < 0) x.y = -x.y;
      if (hk.y < 0) y.y = -y.y;
      const double qt = q[t0 + t];
      s_ab[warp][c][t] = make_double2(qt * (x.x * y.x - x.y * y.y), qt * (x.x * y.y + x.y * y.x));
    }
    __syncwarp();
#pragma unroll 4
    for (int t = 0; t < cnt; ++t) {
      const double2 z = __ldca(tab + (size_t)(t0 + t) * ap.len + ap.off[2] + en.l);
      const double2 w = s_ab[warp][mine][t];
      ac = fma(w.x, z.x, ac);
      bd = fma(w.y, z.y, bd);
      ad = fma(w.x, z.y, ad);
      bc = fma(w.y, z.x, bc);
    }
  }
  red[warp][lane][0] = ac;
  red[warp][lane][1] = bd;
  red[warp][lane][2] = ad;
  red[warp][lane][3] = bc;
  __syncthreads();
  if (warp != 0) return;
  if (e0 + lane >= nentries) return end_after_previous(late);
  for (int w = 1; w < kSf64Warps; ++w) {
    ac += red[w][lane][0];
    bd += red[w][lane][1];
    ad += red[w][lane][2];
    bc += red[w][lane][3];
  }
#pragma unroll
  for (int u = 0; u < 2; ++u) {  // +l, -l
    const int k = u == 0 ? en.kp : en.kn;
    if (k < 0) continue;
    const double w = sqw[k];
    const size_t kcol = 128 * (size_t)(k >> 6) + (k & 63);
    const double re = w * (u == 0 ? ac - bd : ac + bd), im = w * (u == 0 ? ad + bc : bc - ad);
    v[kcol] = add ? v[kcol] + re : re;
    v[kcol + 64] = add ? v[kcol + 64] + im : im;
  }
  end_after_previous(late);
}

// FP64 storage: b^sol_k[f][i] = sum_c A[i][c] v[f][c], two electrode rows a block, whose eight
// warps split the columns, and four frames per grid row (the rows are read once for them).  One
// warp a row left 512 rows on 64 blocks: 90 us against 21.
constexpr int kF64Frames = 4;
constexpr int kF64Rows = 2;

__global__ void __launch_bounds__(256)
k_bsol_kspace_f64(const double* __restrict__ A, int n, int64_t lda, const double* __restrict__ v,
                  int frames, double* __restrict__ bsol, unsigned long long* stamp) {
  __shared__ double red[8][kF64Rows * kF64Frames];
  wait_previous(false);
  stamp_time(stamp);
  v = fresh(v);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row0 = blockIdx.x * kF64Rows;
  const int f0 = blockIdx.y * kF64Frames, nf = min(kF64Frames, frames - f0);
  const double* a[kF64Rows];
#pragma unroll
  for (int i = 0; i < kF64Rows; ++i) a[i] = A + (int64_t)min(row0 + i, n - 1) * lda;
  double acc[kF64Rows][kF64Frames] = {};
#pragma unroll 2
  for (int64_t c = threadIdx.x * 2; c < lda; c += 512) {
    double2 av[kF64Rows];
#pragma unroll
    for (int i = 0; i < kF64Rows; ++i) av[i] = __ldg(reinterpret_cast<const double2*>(a[i] + c));
#pragma unroll
    for (int r = 0; r < kF64Frames; ++r) {
      if (r >= nf) break;
      const double2 vv = __ldca(reinterpret_cast<const double2*>(v + (int64_t)(f0 + r) * lda + c));
#pragma unroll
      for (int i = 0; i < kF64Rows; ++i)
        acc[i][r] = fma(av[i].y, vv.y, fma(av[i].x, vv.x, acc[i][r]));
    }
  }
#pragma unroll
  for (int i = 0; i < kF64Rows; ++i)
#pragma unroll
    for (int r = 0; r < kF64Frames; ++r) {
      if (r >= nf) break;
      double x = acc[i][r];
      for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      if (lane == 0) red[warp][i * kF64Frames + r] = x;
    }
  __syncthreads();
  const int i = threadIdx.x / kF64Frames, r = threadIdx.x % kF64Frames;
  if (i >= kF64Rows || row0 + i >= n || r >= nf) return;
  double x = 0.0;
  for (int w = 0; w < 8; ++w) x += red[w][threadIdx.x];
  bsol[(int64_t)(f0 + r) * n + row0 + i] = x;
}

// Float storage: b^sol_k[f][i] = sum_c A[i][c] v[f][c] over the tail columns (c >= 2 kh), four
// products summed in float and each four into an error-free float pair, plus the head columns
// from float pairs of A and v (products and sums to ~1e-14; A null: the head alone, added to
// bsol).  A block's eight warps are 8 / WS groups of four rows; the WS warps of a group split
// the columns, and a warp takes NF frames at once, in pairs through paired instructions, so
// each float4 of A serves NF frames and each of v four rows.
//
// One frame of a large electrode is bound by reading A (22.3 GB at 12,800 atoms and 217,619
// k-vectors): one warp a row with one load in flight beside the sum's chain reached 4.4 TB/s
// (5.08 ms); four independent rows a warp and the columns split over the block reach
// 6.6 TB/s (3.37 ms).  Many frames are bound by the sums (eleven paired instructions for
// eight products): 512 atoms, 256 frames 791 -> 479 us with the head.  The head in FP64 (1/64 of
// the float rate) took 241 us more there and 778 us at 26,600 atoms and 16 frames, 157 us in
// float pairs.  512 atoms, one frame: 43 -> 9 us in one launch instead of two.
constexpr int kKsWarps = 8;
constexpr int kKsRows = 4;

template <int NF, int WS>
__global__ void __launch_bounds__(kKsWarps * 32, NF == 8 ? 2 : 1)
k_bsol_kspace_f32(const float* __restrict__ A, int64_t lda, const float2* __restrict__ Ahead,
                  int n, int kh, const float* __restrict__ v, const float2* __restrict__ vhead,
                  int frames, double* __restrict__ bsol, int stream,
                  unsigned long long* stamp) {
  constexpr int NP = (NF + 1) / 2;  // frame pairs (one frame fills both halves of one)
  constexpr int NV = kKsRows * 2 * NP;
  __shared__ float2 sm[kKsWarps][NV];
  wait_previous(false);
  stamp_time(stamp);
  v = fresh(v);
  vhead = fresh(vhead);
  bsol = fresh(bsol);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sub = warp % WS;
  const int row0 = (blockIdx.x * (kKsWarps / WS) + warp / WS) * kKsRows;
  const int f0 = blockIdx.y * NF;
  int64_t arow[kKsRows];  // a row past the last repeats it and is not written
#pragma unroll
  for (int i = 0; i < kKsRows; ++i) arow[i] = min(row0 + i, n - 1);
  int frame[2 * NP];
#pragma unroll
  for (int r = 0; r < 2 * NP; ++r) frame[r] = min(f0 + (r < NF ? r : 0), frames - 1);
  float2 hi[kKsRows][NP], lo[kKsRows][NP];
#pragma unroll
  for (int i = 0; i < kKsRows; ++i)
#pragma unroll
    for (int p = 0; p < NP; ++p) hi[i][p] = lo[i][p] = make_float2(0.f, 0.f);
  if (A) {
    for (int64_t c = 2 * (int64_t)kh + (sub * 32 + lane) * 4; c < lda; c += 128 * WS) {
      float a[kKsRows][4];
#pragma unroll
      for (int i = 0; i < kKsRows; ++i) {
        const float4* p = reinterpret_cast<const float4*>(A + arow[i] * lda + c);
        *reinterpret_cast<float4*>(a[i]) = stream ? __ldcs(p) : __ldg(p);
      }
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        float va[4], vb[4];
        *reinterpret_cast<float4*>(va) =
            __ldca(reinterpret_cast<const float4*>(v + frame[2 * p] * lda + c));
        *reinterpret_cast<float4*>(vb) =
            NF == 1 ? *reinterpret_cast<float4*>(va)
                    : __ldca(reinterpret_cast<const float4*>(v + frame[2 * p + 1] * lda + c));
#pragma unroll
        for (int i = 0; i < kKsRows; ++i) {
          float2 s = make_float2(0.f, 0.f);
#pragma unroll
          for (int u = 0; u < 4; ++u)
            s = __ffma2_rn(make_float2(a[i][u], a[i][u]), make_float2(va[u], vb[u]), s);
          pair_add2(hi[i][p], lo[i][p], s);
        }
      }
    }
  }
  // head: two columns a lane
  const int64_t ldh = 2 * (int64_t)kh;
  for (int64_t c = (sub * 32 + lane) * 2; c < ldh; c += 64 * WS) {
    float4 a[kKsRows];  // (hi, lo) of columns c and c + 1
#pragma unroll
    for (int i = 0; i < kKsRows; ++i)
      a[i] = __ldg(reinterpret_cast<const float4*>(Ahead + arow[i] * ldh + c));
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const float4 x = __ldca(reinterpret_cast<const float4*>(vhead + frame[2 * p] * ldh + c));
      const float4 y =
          NF == 1 ? x : __ldca(reinterpret_cast<const float4*>(vhead + frame[2 * p + 1] * ldh + c));
#pragma unroll
      for (int i = 0; i < kKsRows; ++i)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const float ah = u ? a[i].z : a[i].x, al = u ? a[i].w : a[i].y;
          const float2 vh = u ? make_float2(x.z, y.z) : make_float2(x.x, y.x);
          const float2 vl = u ? make_float2(x.w, y.w) : make_float2(x.y, y.y);
          pair_dot2(hi[i][p], lo[i][p], make_float2(ah, ah), make_float2(-ah, -ah),
                    make_float2(al, al), vh, vl);
        }
    }
  }
  // lanes, then the group's warps in order
#pragma unroll
  for (int i = 0; i < kKsRows; ++i)
#pragma unroll
    for (int r = 0; r < NF; ++r) {
      float h = (r & 1) ? hi[i][r >> 1].y : hi[i][r >> 1].x;
      float l = (r & 1) ? lo[i][r >> 1].y : lo[i][r >> 1].x;
#pragma unroll
      for (int o = 16; o; o >>= 1)
        pair_add_pair(h, l, __shfl_xor_sync(0xffffffffu, h, o),
                      __shfl_xor_sync(0xffffffffu, l, o));
      if (lane == 0) sm[warp][i * NF + r] = make_float2(h, l);
    }
  __syncthreads();
  for (int t = threadIdx.x; t < (kKsWarps / WS) * kKsRows * NF; t += kKsWarps * 32) {
    const int g = t / (kKsRows * NF), e = t % (kKsRows * NF);
    const int row = (blockIdx.x * (kKsWarps / WS) + g) * kKsRows + e / NF, f = f0 + e % NF;
    double x = 0.0;
#pragma unroll
    for (int w = 0; w < WS; ++w) x += (double)sm[g * WS + w][e].x + (double)sm[g * WS + w][e].y;
    if (row < n && f < frames) {
      double* dst = bsol + (int64_t)f * n + row;
      *dst = A ? x : *dst + x;
    }
  }
}

// Streamed builds keep no A: b^sol_k[f][i] = sum_{k >= kh} sqrt(W_k) [cos(K.r_i) v_c +
// sin(K.r_i) v_s] with the electrode phases formed on the fly (fixed point, the arithmetic of
// sincos_table); the terms of kDirectBlock consecutive k-vectors are summed in float, and each
// block's sum goes into an error-free float pair (a two-sum), so the rounding of the plain sums
// grows with the block, not with the ~10^5 k-vectors.  One thread per electrode atom and up to
// kDirectFrames frames per block: each phasor is formed once and used for every frame of
// the block; the k-vectors of a chunk and their structure factors are staged in shared
// memory.  Frames go in pairs through paired float instructions (two IEEE results an
// instruction, a - b as fma(b, -1, a)): the values are those of one frame at a time.
//
// Bound by the load unit: a phasor's 16-byte table entry is a random one.  From the 4,096-entry
// table in L1 that took about ten wavefronts a warp (78% of the load unit's time, 2.32 ms at
// 26,600 atoms, 22,700 k-vectors, 16 frames); the first quadrant of it (1,024 entries, the
// others by symmetry: exact swaps and signs) fits shared memory eight times, once for every
// 16-byte bank group, so that the eight lanes of a quarter warp never meet: four wavefronts,
// 1.84 ms.  128 KB of table leave one block of 512 threads an SM.
constexpr int kDirectChunk = 128;
constexpr int kDirectFrames = 16;
constexpr int kDirectBlock = 8;  // divides every chunk: head and table ends are multiples of 16
constexpr int kDirectThreads = 512;
constexpr int kQuadrant = 1024;

struct DirectSmem {
  float4 table[kQuadrant][8];
  // sqrt(W) (v_cos, v_sin) of frames 2 p and 2 p + 1: (c_2p, c_2p+1, s_2p, s_2p+1)
  float4 sv[kDirectChunk][kDirectFrames / 2];
  uint4 sh[kDirectChunk];  // h, k, l
};

__global__ void __launch_bounds__(kDirectThreads, 1)
k_bsol_kspace_direct(const uint32_t* __restrict__ sfix, int n, const int* __restrict__ hkl,
                     const double* __restrict__ sqw, int mpad, int kh,
                     const float4* __restrict__ turn, const float* __restrict__ v, int frames,
                     double* __restrict__ bsol, int nsplit, int64_t split_stride,
                     unsigned long long* stamp) {
  extern __shared__ __align__(16) unsigned char direct_smem[];
  stamp_time(stamp);
  DirectSmem& sm = *reinterpret_cast<DirectSmem*>(direct_smem);
  for (int e = threadIdx.x; e < kQuadrant * 8; e += kDirectThreads)
    sm.table[e >> 3][e & 7] = __ldg(turn + (e >> 3));
  const float4* tab = &sm.table[0][threadIdx.x & 7];
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
  for (int k0 = kbeg; k0 < kend; k0 += kDirectChunk) {
    const int cnt = min(kDirectChunk, kend - k0);
    __syncthreads();
    for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
      const int k = k0 + t;
      sm.sh[t] = make_uint4((uint32_t)hkl[3 * k], (uint32_t)hkl[3 * k + 1],
                            (uint32_t)hkl[3 * k + 2], 0u);
    }
    for (int e = threadIdx.x; e < cnt * (kDirectFrames / 2); e += blockDim.x) {
      const int t = e % kDirectChunk, fp = e / kDirectChunk;
      if (t >= cnt) continue;
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
      sm.sv[t][fp] = val;
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
        const uint4 hk = sm.sh[t];
        const uint32_t ph = hk.x * u0 + hk.y * u1 + hk.z * u2;
        float s0, c0;
        sincos_entry(tab[8 * ((ph >> 20) & (kQuadrant - 1))], ph, &s0, &c0);
        // quadrants 1 and 3 swap; the cosine's sign is set in 1 and 2, the sine's in 2 and 3
        const bool swap = (ph & 0x40000000u) != 0;
        const float cs = __uint_as_float(__float_as_uint(swap ? s0 : c0) ^
                                         ((ph + 0x40000000u) & 0x80000000u));
        const float sn = __uint_as_float(__float_as_uint(swap ? c0 : s0) ^ (ph & 0x80000000u));
        const float2 sn2 = make_float2(sn, sn), cs2 = make_float2(cs, cs);
#pragma unroll
        for (int f = 0; f < kDirectFrames / 2; ++f) {
          const float4 vv = sm.sv[t][f];
          blk[f] = __ffma2_rn(sn2, make_float2(vv.z, vv.w),
                              __ffma2_rn(cs2, make_float2(vv.x, vv.y), blk[f]));
        }
      }
#pragma unroll
      for (int f = 0; f < kDirectFrames / 2; ++f) pair_add2(hi[f], lo[f], blk[f]);
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

// The tail k-vectors [kh, m) of the table hkl in pairs with equal h, k and consecutive l (a
// k-vector without a partner alone, k1 = -1), and the table's padding [m, mpad) alone.
std::vector<SfPair> sf_pairs(const std::vector<int>& hkl, int m, int mpad, int kh) {
  int lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
  for (int k = 0; k < m; ++k)
    for (int d = 0; d < 3; ++d) {
      lo[d] = std::min(lo[d], hkl[3 * (size_t)k + d]);
      hi[d] = std::max(hi[d], hkl[3 * (size_t)k + d]);
    }
  const size_t nl = hi[2] - lo[2] + 1, nk = hi[1] - lo[1] + 1, nh = hi[0] - lo[0] + 1;
  std::vector<int> at(nh * nk * nl, -1);  // tail k-vector at (h, k, l)
  for (int k = kh; k < m; ++k)
    at[((hkl[3 * (size_t)k] - lo[0]) * nk + (hkl[3 * (size_t)k + 1] - lo[1])) * nl +
       (hkl[3 * (size_t)k + 2] - lo[2])] = k;
  std::vector<SfPair> out;
  out.reserve((m - kh) / 2 + (m - kh) / 16 + 64);
  for (size_t c = 0; c < nh * nk; ++c) {
    const int h = (int)(c / nk) + lo[0], k = (int)(c % nk) + lo[1];
    for (size_t l = 0; l < nl; ++l) {
      const int k0 = at[c * nl + l];
      if (k0 < 0) continue;
      const int k1 = l + 1 < nl ? at[c * nl + l + 1] : -1;
      out.push_back({h, k, (int)l + lo[2], k0, k1});
      if (k1 >= 0) ++l;
    }
  }
  for (int k = std::max(kh, m); k < mpad; ++k) out.push_back({0, 0, 0, k, -1});
  return out;
}

// The k-vectors of the table hkl [0, m) in entries of equal h, k and opposite l, column by column
// ((h, k) pairs), with |l| running up within a column.
std::vector<SfEntry> sf_entries(const std::vector<int>& hkl, int m) {
  int lo[2] = {0, 0}, hi[2] = {0, 0}, lmax = 0;
  for (int k = 0; k < m; ++k) {
    for (int d = 0; d < 2; ++d) {
      lo[d] = std::min(lo[d], hkl[3 * (size_t)k + d]);
      hi[d] = std::max(hi[d], hkl[3 * (size_t)k + d]);
    }
    lmax = std::max(lmax, std::abs(hkl[3 * (size_t)k + 2]));
  }
  const size_t nk = hi[1] - lo[1] + 1, nc = (hi[0] - lo[0] + 1) * nk, nl = lmax + 1;
  std::vector<int> at(2 * nc * nl, -1);  // places of (h, k, l) and (h, k, -l)
  for (int k = 0; k < m; ++k) {
    const int* p = &hkl[3 * (size_t)k];
    at[2 * (((p[0] - lo[0]) * nk + (p[1] - lo[1])) * nl + std::abs(p[2])) + (p[2] < 0)] = k;
  }
  std::vector<SfEntry> out;
  out.reserve(m / 2 + m / 16 + 64);
  int col = -1;
  for (size_t c = 0; c < nc; ++c) {
    bool first = true;
    for (size_t l = 0; l < nl; ++l) {
      const int kp = at[2 * (c * nl + l)], kn = at[2 * (c * nl + l) + 1];
      if (kp < 0 && kn < 0) continue;
      if (first) ++col;
      first = false;
      out.push_back({(int)(c / nk) + lo[0], (int)(c % nk) + lo[1], (int)l, col, kp, kn});
    }
  }
  return out;
}

void launch_axis_phasors(const double* xyz, const uint32_t* sfix, int64_t count,
                         const double L[3], const AxisPhasors& ap, double2* out,
                         cudaStream_t s) {
  const int blocks = (int)std::min<int64_t>((count * ap.len + 127) / 128, 16384);
  launch_next(k_axis_phasors, dim3(blocks), 128, 0, s, xyz, sfix, count, L[0], L[1], L[2], ap,
              out);
}

void launch_ion_structure_factor(bool fp64, const double2* axis, const AxisPhasors& ap,
                                 const uint32_t* sion, int64_t coord_stride,
                                 const double* ion_q, int64_t charge_stride, int frames, int n_ion,
                                 bool add, const SfList& kl, const int* hkl,
                                 const double* sqw, int m, int mpad, int kh, const void* turn,
                                 void* v, void* vhead, int sms, bool late,
                                 unsigned long long* stamp, cudaStream_t s) {
  if (fp64) {
    launch_next(k_ion_sf_f64, dim3(std::max(1, (kl.entries + 31) / 32), frames), kSf64Warps * 32, 0,
                s, axis, ap, coord_stride, ion_q, charge_stride, n_ion, add, (const SfEntry*)kl.list,
                kl.entries, sqw, m, mpad, (double*)v, late, stamp);
  } else {
    // warps of a block split the ions until the chip's warps are busy (24 resident an SM),
    // each with at least four blocks of eight ions, and, to even out the last wave, up to four
    // times as far where a share keeps 512 points (16 frames of 5,000 ions, 26,600 atoms:
    // 1,607 -> 1,450 us; 2,000 ions of one frame split further 337 -> 345)
    const SfPair* pairs = (const SfPair*)kl.list;
    const int npairs = kl.entries;
    const int groups = (npairs + 31) / 32;
    int shares = 1;
    while (shares < kSfWarps) {
      const int64_t warps = (int64_t)groups * frames * shares;
      if (!(warps < 24 * (int64_t)sms && n_ion >= 64 * shares) &&
          !(warps < 96 * (int64_t)sms && n_ion >= 1024 * shares))
        break;
      shares *= 2;
    }
    const int per = 32 * (kSfWarps / shares), hb = (kh + 31) / 32;
    launch_next(k_ion_sf_f32, dim3(hb + (npairs + per - 1) / per, frames), kSfWarps * 32, 0, s, sion,
                coord_stride, ion_q, n_ion, pairs, npairs, hkl, sqw, mpad, kh, shares, hb,
                (const float4*)turn, (float*)v, (float2*)vhead, late, stamp);
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

// Shares of the k range for the direct sum: the atom blocks of kDirectFrames-frame groups (one
// resident an SM) times the shares fill whole waves of `sms` SMs best (a larger count only
// where it fills 2% more of the last wave; at least eight chunks a share, against the 128 KB
// of table a block writes first).
int bsol_direct_splits(int n, int frames, int mpad, int kh, int sms) {
  const int64_t blocks = (int64_t)((n + kDirectThreads - 1) / kDirectThreads) *
                         ((frames + kDirectFrames - 1) / kDirectFrames);
  const int nch = (mpad - kh + kDirectChunk - 1) / kDirectChunk;
  int best = 1;
  double best_eff = -1.0;
  for (int sp = 1; sp <= std::min(24, std::max(1, nch / 8)); ++sp) {
    const int64_t units = blocks * sp, waves = (units + sms - 1) / sms;
    const double eff = (double)units / (double)(waves * sms);
    if (eff > best_eff + 0.02) {
      best_eff = eff;
      best = sp;
    }
  }
  return best;
}

namespace {

template <int NF, int WS>
void launch_kspace_f32(const float* A, int64_t lda, const float2* Ahead, int n, int kh,
                       const float* v, const float2* vhead, int frames, double* bsol,
                       unsigned long long* stamp, cudaStream_t s) {
  constexpr int kRows = kKsRows * (kKsWarps / WS);
  const int groups = (frames + NF - 1) / NF;
  // A larger than half of L2 is read past it once (v and the sums' operands stay)
  const int stream = A && (int64_t)n * lda * (int64_t)sizeof(float) > (64ll << 20);
  for (int g0 = 0; g0 < groups; g0 += 65535) {
    const int f0 = g0 * NF;
    launch_next(k_bsol_kspace_f32<NF, WS>, dim3((n + kRows - 1) / kRows, std::min(groups - g0, 65535)),
                kKsWarps * 32, 0, s, A, lda, Ahead, n, kh, v + f0 * lda,
                vhead + (int64_t)f0 * 2 * kh, frames - f0, bsol + (int64_t)f0 * n, stream,
                g0 == 0 ? stamp : nullptr);
  }
}

// Eight frames at a time; fewer frames in one pass of the next larger size.  Rows share their
// frames' v within a block (two warps a group) where that leaves two blocks an SM.
void launch_kspace_frames(const float* A, int64_t lda, const float2* Ahead, int n, int kh,
                          const float* v, const float2* vhead, int frames, double* bsol,
                          int sms, unsigned long long* stamp, cudaStream_t s) {
  if (frames == 1)
    launch_kspace_f32<1, 8>(A, lda, Ahead, n, kh, v, vhead, frames, bsol, stamp, s);
  else if (frames == 2)
    launch_kspace_f32<2, 8>(A, lda, Ahead, n, kh, v, vhead, frames, bsol, stamp, s);
  else if (frames <= 4)
    launch_kspace_f32<4, 8>(A, lda, Ahead, n, kh, v, vhead, frames, bsol, stamp, s);
  else if ((int64_t)((n + 15) / 16) * ((frames + 7) / 8) >= 2 * (int64_t)sms)
    launch_kspace_f32<8, 2>(A, lda, Ahead, n, kh, v, vhead, frames, bsol, stamp, s);
  else
    launch_kspace_f32<8, 8>(A, lda, Ahead, n, kh, v, vhead, frames, bsol, stamp, s);
}

}  // namespace

// b^sol_k = A v: in float storage the head k-vectors (the heaviest weights) are contracted in
// float pairs against a float-pair copy of their operand columns.  Without A (a streamed
// build) the float part is the direct sum over the tail k-vectors.
void launch_bsol_kspace(bool fp64, const void* A, const void* Ahead, int n, int mpad, int kh,
                        const void* v, const void* vhead, int frames, double* bsol,
                        const uint32_t* sfix, const int* hkl, const double* sqw,
                        const void* turn, int nsplit, double* split_part, int sms,
                        unsigned long long* stamp, cudaStream_t s) {
  const int64_t lda = 2 * (int64_t)mpad;
  if (fp64) {
    const int groups = (frames + kF64Frames - 1) / kF64Frames;
    for (int g0 = 0; g0 < groups; g0 += 65535) {
      const int f0 = kF64Frames * g0;
      launch_next(k_bsol_kspace_f64, dim3((n + kF64Rows - 1) / kF64Rows, std::min(groups - g0, 65535)),
                  256, 0, s, (const double*)A, n, lda, (const double*)v + f0 * lda, frames - f0,
                  bsol + (int64_t)f0 * n, g0 == 0 ? stamp : nullptr);
    }
    return;
  }
  if (!A) {
    const int fgroups = (frames + kDirectFrames - 1) / kDirectFrames;
    const int sp = split_part ? nsplit : 1;
    const int64_t stride = (int64_t)frames * n;  // between shares
    double* dst = sp > 1 ? split_part : bsol;
    cudaFuncSetAttribute(k_bsol_kspace_direct, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sizeof(DirectSmem));  // a failure shows at the launch
    for (int g0 = 0; g0 < fgroups; g0 += 65535) {
      const int f0 = g0 * kDirectFrames;
      const int nblk = (n + kDirectThreads - 1) / kDirectThreads;
      (k_bsol_kspace_direct<<<dim3(sp * nblk, std::min(fgroups - g0, 65535)), kDirectThreads,
                              sizeof(DirectSmem), s>>>(
           sfix, n, hkl, sqw, mpad, kh, (const float4*)turn, (const float*)v + f0 * lda,
           frames - f0, dst + (int64_t)f0 * n, sp, stride, g0 == 0 ? stamp : nullptr),
       note_launch());
    }
    if (sp > 1)
      (k_sum_splits<<<(int)std::min<int64_t>((stride + 255) / 256, 8192), 256, 0, s>>>(
           split_part, sp, stride, stride, bsol),
       note_launch());
    if (kh == 0) return;
  }
  launch_kspace_frames((const float*)A, lda, (const float2*)Ahead, n, kh, (const float*)v,
                       (const float2*)vhead, frames, bsol, sms, A ? stamp : nullptr, s);
}

}  // namespace cpm
