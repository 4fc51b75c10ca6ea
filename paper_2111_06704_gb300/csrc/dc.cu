// PCG-DC preconditioner (Sec. III B 2, steps 1-3; Eq. 36).
//
// For every electrode atom tau: its neighbours j with |r_tau - r_j| <= r_cut (minimum
// image, tau included, sorted by index); the local matrix M_tau of Eq. 36 over them;
// column tau of M_tau^-1, i.e. the solution of M_tau x = e_tau, by Gaussian elimination
// with partial pivoting in FP64 shared memory (one block per atom).  The column is
// stored as P[j, tau] for the neighbours j; a transpose pass re-files it by row so the
// apply z_j = sum_tau P[j, tau] r_tau is a gather.
#include <math.h>

#include <algorithm>
#include <vector>

#include "cpm_internal.cuh"

namespace cpm {

namespace {

constexpr int kMaxLocal = 160;  // largest neighbourhood held in shared memory

__device__ __forceinline__ double min_image(double d, double L) { return d - L * rint(d / L); }

__device__ __forceinline__ double dist2(const double* a, const double* b, double lx, double ly,
                                        double lz) {
  double dx = min_image(a[0] - b[0], lx), dy = min_image(a[1] - b[1], ly),
         dz = min_image(a[2] - b[2], lz);
  return dx * dx + dy * dy + dz * dz;
}

// One warp per atom: count (fill == 0) or list (fill == 1) its neighbours in index order
// (r <= r_cut, or r < r_cut with strict).
// The candidates of a block are staged as float positions; the float minimum-image
// distance decides every pair outside a band of +-0.01 A^2 around r_cut^2 (float
// positions of a box below 1e4 A are off by < 1e-3 A, so the band is ample), and the
// pairs inside it are decided by the FP64 distance, as the definition asks.  The float
// constants come from the host (a constant formed from the FP64 parameters could be
// re-formed inside the loop, at 1/64 of the float rate).
constexpr int kNbrWarps = 8;
constexpr int kNbrStage = 1024;

struct NbrFloat {
  float L[3], inv[3];  // box edges and their reciprocals
  float lo2, hi2;      // r_cut^2 -+ 0.01: the band decided in FP64
};

__global__ void __launch_bounds__(kNbrWarps * 32)
k_neighbours(const double* __restrict__ xyz, int n, double lx, double ly, double lz,
             double rc2, const NbrFloat nf, int* __restrict__ cnt,
             const int64_t* __restrict__ off, int* __restrict__ idx, int fill, int strict) {
  __shared__ float4 sp[kNbrStage];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = blockIdx.x * kNbrWarps + warp;
  const bool live = t < n;
  const float Lx = nf.L[0], Ly = nf.L[1], Lz = nf.L[2];
  const float ix = nf.inv[0], iy = nf.inv[1], iz = nf.inv[2];
  const float lo2 = nf.lo2, hi2 = nf.hi2;
  float tx = 0.f, ty = 0.f, tz = 0.f;
  if (live) {
    tx = (float)xyz[3 * t];
    ty = (float)xyz[3 * t + 1];
    tz = (float)xyz[3 * t + 2];
  }
  int c = 0;
  for (int base = 0; base < n; base += kNbrStage) {
    const int cj = min(kNbrStage, n - base);
    __syncthreads();
    for (int e = threadIdx.x; e < cj; e += blockDim.x)
      sp[e] = make_float4((float)xyz[3 * (base + e)], (float)xyz[3 * (base + e) + 1],
                          (float)xyz[3 * (base + e) + 2], 0.f);
    __syncthreads();
    if (!live) continue;
    for (int jj = 0; jj < cj; jj += 32) {
      const int j = base + jj + lane;
      bool in = false;
      if (jj + lane < cj) {
        const float4 pj = sp[jj + lane];
        float dx = pj.x - tx, dy = pj.y - ty, dz = pj.z - tz;
        dx -= Lx * rintf(dx * ix);
        dy -= Ly * rintf(dy * iy);
        dz -= Lz * rintf(dz * iz);
        const float r2 = dx * dx + dy * dy + dz * dz;
        if (r2 < lo2) in = true;
        else if (r2 <= hi2) {
          const double d2 = dist2(xyz + 3 * t, xyz + 3 * j, lx, ly, lz);
          in = strict ? d2 < rc2 : d2 <= rc2;
        }
      }
      const unsigned m = __ballot_sync(0xffffffffu, in);
      if (fill && in) idx[off[t] + c + __popc(m & ((1u << lane) - 1u))] = j;
      c += __popc(m);
    }
  }
  if (!fill && live && lane == 0) cnt[t] = c;
}

void launch_neighbours(const double* xyz, int n, const double* L, double rc2, int* cnt,
                       const int64_t* off, int* idx, int fill, int strict, cudaStream_t s) {
  NbrFloat nf;
  for (int u = 0; u < 3; ++u) {
    nf.L[u] = (float)L[u];
    nf.inv[u] = (float)(1.0 / L[u]);
  }
  nf.lo2 = (float)rc2 - 0.01f;
  nf.hi2 = (float)rc2 + 0.01f;
  const int blocks = (n + kNbrWarps - 1) / kNbrWarps;
  (k_neighbours<<<blocks, kNbrWarps * 32, 0, s>>>(xyz, n, L[0], L[1], L[2], rc2, nf, cnt, off,
                                                   idx, fill, strict),
   note_launch());
}

// The off-diagonal value of Eq. 36 for every pattern entry (j, j'): (erfc(g r) -
// erfc(g r_cut)) / r, zero for the atom itself and at r = r_cut.  Every local matrix
// M_tau only holds pairs within r_cut of each other, i.e. pattern entries, so the FP64
// erfc runs once per entry instead of once per entry of every local matrix.
// One warp a row of the pattern (one thread a row, ~140 erfc in a chain, took 446 us at 800
// atoms, 38 us so).
__global__ void k_dc_pairs(const double* __restrict__ xyz, int n, double lx, double ly,
                           double lz, double g, double rcut, const int64_t* __restrict__ off,
                           const int* __restrict__ idx, double* __restrict__ val) {
  const int j = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  if (j >= n) return;
  const double erfc_rc = erfc(g * rcut);
  const double rc2 = rcut * rcut;
  for (int64_t e = off[j] + (threadIdx.x & 31); e < off[j + 1]; e += 32) {
    const int k = idx[e];
    double v = 0.0;
    if (k != j) {
      const double r2 = dist2(xyz + 3 * j, xyz + 3 * k, lx, ly, lz);
      if (r2 < rc2) {
        const double r = sqrt(r2);
        v = (erfc(g * r) - erfc_rc) / r;
      }
    }
    val[e] = v;
  }
}

// Column tau of M_tau^-1 (Eq. 36), written to pcol[off[tau] .. off[tau+1]).  One block
// per atom.  The symmetric local matrix is made of the pattern's FP64 pair values: a pair of
// tau's neighbours closer than r_cut is an entry of both their pattern rows, and a warp walks a
// neighbour's row, coalesced, and finds each entry's position in tau's list, held in shared
// memory, by binary search.  A float copy is factored P M = L U with partial pivoting (FP64
// runs at 1/64 of the float rate here, and the factorisation is m^3 / 3 multiply-adds), and the
// solution is refined against the FP64 matrix: x += (LU)^-1 P (e_tau - M x), residuals in
// FP64.  Each step shrinks the error by about kappa(M) 2^-24 (~1e-5 here), so the error
// left after adding a correction d is about that times |d|: refinement stops once
// |d| <= 1e-9 |x| (error ~1e-13 even at kappa(M) 2^-24 = 1e-4; typically after the
// second correction).
//
// The chains in k bind it: m pivot steps, and two triangular solves of m steps for each
// correction.  Eight warps a block or more (32 an SM) share the row updates; a step's update
// leaves the next step's pivot candidates behind, a barrier a step where no rows are exchanged;
// the row multipliers come from one load a warp; and the solves keep the vector in one warp's
// registers.  Every element of the factors and of
// the vectors is one thread's chain in k, whatever the split.  12,800 atoms, neighbourhoods of
// 79: 8.2 ms with four warps, three barriers a step and the vectors in shared memory, 4.3 ms so (4 or
// 16 warps a block: 5.2, 6.4 ms); issue 55%, FP64 residuals a quarter of the FP64 pipe.
constexpr int kDcMaxThreads = 512;
constexpr int kDcMaxRefine = 6;

__device__ __forceinline__ int sym_index(int a, int b, int m) {  // packed upper, a <= b
  return a * m - (a * (a - 1)) / 2 + (b - a);
}

// shared memory of k_dc_local for a neighbourhood of m atoms
size_t dc_local_smem(int m) {
  return (size_t)m * (m + 1) / 2 * sizeof(double) + 2 * (size_t)m * sizeof(double) +
         (size_t)m * (m + 1) * sizeof(float) + 2 * (size_t)m * sizeof(int);
}

// SEGS: 32-element segments of the longest row
template <int SEGS>
__global__ void __launch_bounds__(kDcMaxThreads, 2)
k_dc_local(const double* __restrict__ alpha, const int64_t* __restrict__ off,
           const int* __restrict__ idx, const double* __restrict__ pval,
           double* __restrict__ pcol, int* __restrict__ status) {
  extern __shared__ double sm[];
  const int warps = blockDim.x >> 5;
  const int tau = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t o = off[tau];
  const int m = (int)(off[tau + 1] - o);
  const int ld = m + 1;                        // float row stride
  double* S = sm;                              // packed upper triangle of M (FP64)
  double* x = S + (size_t)m * (m + 1) / 2;     // solution (FP64)
  double* r = x + m;                           // residual (FP64)
  float* F = reinterpret_cast<float*>(r + m);  // [m][ld]: L (unit, below) and U
  int* perm = reinterpret_cast<int*>(F + (size_t)m * ld);  // row of M at each row of L U
  int* list = perm + m;                        // tau's neighbours (ascending)
  __shared__ uint2 cand[2][kDcMaxThreads / 32];  // pivot candidates: |value|'s bits, row
  __shared__ int s_pos, s_done;
  for (int e = threadIdx.x; e < m * (m + 1) / 2; e += blockDim.x) S[e] = 0.0;
  for (int e = threadIdx.x; e < m * ld; e += blockDim.x) F[e] = 0.f;
  for (int a = threadIdx.x; a < m; a += blockDim.x) {
    const int j = idx[o + a];
    list[a] = j;
    perm[a] = a;
    if (j == tau) s_pos = a;
  }
  __syncthreads();
  for (int a = warp; a < m; a += warps) {
    const int ja = list[a];
    for (int64_t e = off[ja] + lane; e < off[ja + 1]; e += 32) {
      const int jb = idx[e];
      int lo = a + 1, hi = m;  // position of jb in tau's list, if there and after a
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (list[mid] < jb) lo = mid + 1;
        else hi = mid;
      }
      if (lo < m && list[lo] == jb) {
        const double v = pval[e];
        S[sym_index(a, lo, m)] = v;
        F[a * ld + lo] = F[lo * ld + a] = (float)v;
      }
    }
    if (lane == 0) {
      const double al = alpha[ja], v = isinf(al) ? 0.0 : 0.7978845608028654 * al;  // sqrt(2/pi)
      S[sym_index(a, a, m)] = v;
      F[a * ld + a] = (float)v;
    }
  }
  __syncthreads();
  // ---- P M = L U in float, partial pivoting (largest, then first), whole rows exchanged -----
  auto bits = [](float v) { v = fabsf(v); return v == v ? __float_as_uint(v) : 0u; };
  // lane l looks after the warp's l-th row past k (never more than 32: sixteen warps take up to
  // kMaxLocal atoms, four at most 96)
  auto candidate = [&](int a, int k) {  // the warp's largest of column k, rows a of its lanes
    const unsigned v = a < m ? bits(F[a * ld + k]) : 0u;
    const unsigned mx = __reduce_max_sync(0xffffffffu, v);
    const int bi = __reduce_min_sync(0xffffffffu, v == mx ? a : INT_MAX);
    if (lane == 0) cand[k & 1][warp] = make_uint2(mx, (unsigned)bi);
  };
  candidate(warp + warps * lane, 0);
  __syncthreads();
  for (int k = 0; k < m; ++k) {
    const uint2 c = lane < warps ? cand[k & 1][lane] : make_uint2(0u, (unsigned)INT_MAX);
    const unsigned mx = __reduce_max_sync(0xffffffffu, c.x);
    const int pv = __reduce_min_sync(0xffffffffu, c.x == mx ? (int)c.y : INT_MAX);
    if (mx == 0u) {
      if (threadIdx.x == 0) atomicExch(status, 1);
      return;  // singular local matrix (whole block leaves together)
    }
    if (pv != k) {
      for (int b = threadIdx.x; b < m; b += blockDim.x) {
        const float t = F[k * ld + b];
        F[k * ld + b] = F[pv * ld + b];
        F[pv * ld + b] = t;
      }
      if (threadIdx.x == 0) {
        const int t = perm[k];
        perm[k] = perm[pv];
        perm[pv] = t;
      }
      __syncthreads();
    }
    const float inv = 1.f / F[k * ld + k];
    const int a0 = k + 1 + warp, al = a0 + warps * lane;
    const float fl = al < m ? F[al * ld + k] * inv : 0.f;
    float u[SEGS];  // row k of U
    bool on[SEGS];
#pragma unroll
    for (int i = 0; i < SEGS; ++i) {
      const int b = lane + 32 * i;
      on[i] = b > k && b < m;
      u[i] = on[i] ? F[k * ld + b] : 0.f;
    }
    float* Fa = F + a0 * ld + lane;
    for (int a = a0, l = 0; a < m; a += warps, ++l, Fa += warps * ld) {
      const float f = __shfl_sync(0xffffffffu, fl, l);
#pragma unroll
      for (int i = 0; i < SEGS; ++i) {
        if (32 * i + 31 <= k) continue;
        if (on[i]) Fa[32 * i] = fmaf(-f, u[i], Fa[32 * i]);
      }
    }
    __syncwarp();
    if (al < m) F[al * ld + k] = fl;
    if (k + 1 < m) candidate(al, k + 1);
    __syncthreads();
  }
  // ---- x = 0, r = e_tau; x += (LU)^-1 P r; r = e_tau - M x (FP64) ------------------------
  for (int a = threadIdx.x; a < m; a += blockDim.x) {
    x[a] = 0.0;
    r[a] = a == s_pos ? 1.0 : 0.0;
  }
  if (threadIdx.x == 0) s_done = 0;
  __syncthreads();
  for (int it = 0; it < kDcMaxRefine && !s_done; ++it) {
    if (warp == 0) {
      // element a = lane + 32 i of the vector in y[i]; lanes past m compute and are not read
      float y[SEGS];
      const float* Fr[SEGS];
#pragma unroll
      for (int i = 0; i < SEGS; ++i) {
        const int a = min(lane + 32 * i, m - 1);
        y[i] = (float)r[perm[a]];
        Fr[i] = F + a * ld;
      }
#pragma unroll
      for (int ib = 0; ib < SEGS; ++ib) {  // forward: unit lower L
        const int n = min(32, m - 32 * ib);
#pragma unroll 4
        for (int kk = 0; kk < n; ++kk) {
          const int k = 32 * ib + kk;
          const float yk = __shfl_sync(0xffffffffu, y[ib], kk);
#pragma unroll
          for (int i = ib; i < SEGS; ++i) {
            const float t = fmaf(-Fr[i][k], yk, y[i]);
            if (i > ib || lane > kk) y[i] = t;
          }
        }
      }
#pragma unroll
      for (int ib = SEGS - 1; ib >= 0; --ib) {  // back: U
        const int n = min(32, m - 32 * ib);
#pragma unroll 4
        for (int kk = n - 1; kk >= 0; --kk) {
          const int k = 32 * ib + kk;
          const float yk = __shfl_sync(0xffffffffu, y[ib], kk) / F[k * ld + k];
#pragma unroll
          for (int i = 0; i <= ib; ++i) {
            const float t = fmaf(-Fr[i][k], yk, y[i]);
            if (i < ib || lane < kk) y[i] = t;
          }
          if (lane == kk) y[ib] = yk;
        }
      }
      double dmax = 0.0, xmax = 0.0;
#pragma unroll
      for (int i = 0; i < SEGS; ++i) {
        const int a = lane + 32 * i;
        if (a >= m) continue;
        x[a] += (double)y[i];
        dmax = fmax(dmax, fabs((double)y[i]));
        xmax = fmax(xmax, fabs(x[a]));
      }
      for (int sh = 16; sh; sh >>= 1) {
        dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, sh));
        xmax = fmax(xmax, __shfl_xor_sync(0xffffffffu, xmax, sh));
      }
      if (lane == 0 && dmax <= 1e-9 * xmax) s_done = 1;
    }
    __syncthreads();
    if (s_done) break;
    for (int a = warp; a < m; a += warps) {  // r = e_tau - M x, one warp per row
      double s = 0.0;
      for (int b = lane; b < m; b += 32)
        s += S[a <= b ? sym_index(a, b, m) : sym_index(b, a, m)] * x[b];
      for (int sh = 16; sh; sh >>= 1) s += __shfl_xor_sync(0xffffffffu, s, sh);
      if (lane == 0) r[a] = (a == s_pos ? 1.0 : 0.0) - s;
    }
    __syncthreads();
  }
  for (int a = threadIdx.x; a < m; a += blockDim.x) pcol[o + a] = x[a];
}

// prow[off[j] + position of tau in j's list] = pcol[off[tau] + a] - shift, j = idx[off[tau] + a]
__global__ void k_dc_transpose(int n, const int64_t* __restrict__ off, const int* __restrict__ idx,
                               const double* __restrict__ pcol, double shift,
                               double* __restrict__ prow) {
  const int tau = blockIdx.x;
  for (int64_t e = off[tau] + threadIdx.x; e < off[tau + 1]; e += blockDim.x) {
    const int j = idx[e];
    int64_t lo = off[j], hi = off[j + 1];
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (idx[mid] < tau) lo = mid + 1;
      else hi = mid;
    }
    if (lo < off[j + 1] && idx[lo] == tau) prow[lo] = pcol[e] - shift;
  }
}

__global__ void k_sum_blocks(const double* __restrict__ v, int64_t len, double* __restrict__ part) {
  __shared__ double sm[32];
  double s = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len;
       i += (int64_t)gridDim.x * blockDim.x)
    s += v[i];
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = threadIdx.x < (blockDim.x >> 5) ? sm[threadIdx.x] : 0.0;
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
  }
}

}  // namespace

// Sum of a device vector, deterministic (fixed block partials, host sum in order).
int device_sum(Ctx* c, const double* v, int64_t len, double* out) {
  const int blocks = 256;
  Buf tmp;
  if (int rc = buf_alloc(c, &tmp, blocks * sizeof(double))) return rc;
  (k_sum_blocks<<<blocks, 256, 0, c->stream>>>(v, len, (double*)tmp.ptr), note_launch());
  std::vector<double> h(blocks);
  int rc = cuda_check(c, cudaMemcpyAsync(h.data(), tmp.ptr, blocks * sizeof(double),
                                         cudaMemcpyDeviceToHost, c->stream), "sum copy");
  if (!rc) rc = cuda_check(c, cudaStreamSynchronize(c->stream), "sum sync");
  buf_free(c, &tmp);
  if (rc) return rc;
  double s = 0.0;
  for (double x : h) s += x;
  *out = s;
  return CPM_OK;
}

// Builds the neighbour pattern and the row form of P (without p_gap).
int build_dc_preconditioner(Ctx* c) {
  const int n = c->n;
  const double* L = c->p.box;
  const double rc = c->p.rcut_dc;
  if (!(rc > 0.0) || 2.0 * rc >= std::min(L[0], std::min(L[1], L[2])))
    return set_err(c, CPM_EINVAL, "rcut_dc must be positive and below half of every box edge");
  cudaStream_t s = c->stream;
  // workspace kept by the context (buf_reserve): the counts, the local solutions, a flag
  Buf &cnt = c->dc_cnt, &pcol = c->dc_pcol, &status = c->dc_status;
  if (int rc2 = buf_reserve(c, &cnt, (size_t)n * sizeof(int))) return rc2;
  launch_neighbours((const double*)c->xyz.ptr, n, L, rc * rc, (int*)cnt.ptr, nullptr, nullptr,
                    0, 0, s);
  std::vector<int> hc(n);
  int st = cuda_check(c, cudaMemcpyAsync(hc.data(), cnt.ptr, n * sizeof(int),
                                         cudaMemcpyDeviceToHost, s), "dc counts");
  if (!st) st = cuda_check(c, cudaStreamSynchronize(s), "dc counts sync");
  if (st) return st;
  std::vector<int64_t> off(n + 1, 0);
  int mx = 0;
  for (int i = 0; i < n; ++i) {
    off[i + 1] = off[i] + hc[i];
    mx = std::max(mx, hc[i]);
  }
  if (mx > kMaxLocal)
    return set_err(c, CPM_EINVAL, "PCG-DC neighbourhood larger than 160 atoms; lower rcut_dc");
  c->nnz = off[n];
  if ((st = buf_reserve(c, &c->nbr_off, (n + 1) * sizeof(int64_t)))) return st;
  if ((st = buf_reserve(c, &c->nbr_idx, c->nnz * sizeof(int)))) return st;
  if ((st = buf_reserve(c, &c->prow, c->nnz * sizeof(double)))) return st;
  if ((st = buf_reserve(c, &pcol, c->nnz * sizeof(double)))) return st;
  if ((st = buf_reserve(c, &status, sizeof(int)))) return st;
  st = cuda_check(c, cudaMemcpyAsync(c->nbr_off.ptr, off.data(), (n + 1) * sizeof(int64_t),
                                     cudaMemcpyHostToDevice, s), "dc offsets");
  if (!st) st = cuda_check(c, cudaMemsetAsync(status.ptr, 0, sizeof(int), s), "dc status");
  if (!st) {
    launch_neighbours((const double*)c->xyz.ptr, n, L, rc * rc, nullptr,
                      (const int64_t*)c->nbr_off.ptr, (int*)c->nbr_idx.ptr, 1, 0, s);
    const size_t smem = dc_local_smem(mx);
    // about 32 warps an SM, at least four and at most sixteen a block
    const int fit = (int)(((size_t)227 << 10) / (smem + 1024));
    const int warps = fit <= 2 ? 16 : fit <= 5 ? 8 : 4;
    auto local = mx <= 32   ? k_dc_local<1>
                 : mx <= 64 ? k_dc_local<2>
                 : mx <= 96 ? k_dc_local<3>
                 : mx <= 128 ? k_dc_local<4>
                             : k_dc_local<kMaxLocal / 32>;
    st = cuda_check(c, cudaFuncSetAttribute(local, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)smem), "dc smem");
    if (!st) {
      // pair values of the pattern, held in prow until the transpose overwrites it
      (k_dc_pairs<<<(n + 3) / 4, 128, 0, s>>>((const double*)c->xyz.ptr, n, L[0], L[1],
                                                  L[2], c->p.g_dc, rc,
                                                  (const int64_t*)c->nbr_off.ptr,
                                                  (const int*)c->nbr_idx.ptr,
                                                  (double*)c->prow.ptr), note_launch());
      (local<<<n, warps * 32, smem, s>>>((const double*)c->alpha.ptr,
                                              (const int64_t*)c->nbr_off.ptr,
                                              (const int*)c->nbr_idx.ptr,
                                              (const double*)c->prow.ptr, (double*)pcol.ptr,
                                              (int*)status.ptr), note_launch());
      (k_dc_transpose<<<n, 128, 0, s>>>(n, (const int64_t*)c->nbr_off.ptr,
                                       (const int*)c->nbr_idx.ptr, (const double*)pcol.ptr, 0.0,
                                       (double*)c->prow.ptr), note_launch());
      st = cuda_check(c, cudaGetLastError(), "dc kernels");
    }
  }
  int hs = 0;
  if (!st) st = cuda_check(c, cudaMemcpyAsync(&hs, status.ptr, sizeof(int),
                                              cudaMemcpyDeviceToHost, s), "dc status copy");
  if (!st) st = cuda_check(c, cudaStreamSynchronize(s), "dc sync");
  if (st) return st;
  if (hs) return set_err(c, CPM_EINVAL, "a PCG-DC local matrix is singular");
  return CPM_OK;
}

// P[j][tau] = (E^-1)_{j tau} on the pattern, from the columns E^-1 e_tau (column-major,
// X[tau * n + j]); one block per row j.
__global__ void k_gather_inverse(int n, const int64_t* __restrict__ off,
                                 const int* __restrict__ idx, const double* __restrict__ X,
                                 double* __restrict__ prow) {
  const int j = blockIdx.x;
  for (int64_t e = off[j] + threadIdx.x; e < off[j + 1]; e += blockDim.x)
    prow[e] = X[(int64_t)idx[e] * n + j];
}

// PCG-Normal / PCG-Full (Sec. III B 2, Fig. 6a): the pattern of the pairs within the
// cutoff (minimum image; r < rcut_dc for Normal, r <= rcut_real for Full) and the entries
// of E^-1 on it, from the n columns E^-1 e_j solved by the context's PCG with the Jacobi
// preconditioner to 1e-10.  No p_gap fill.  n <= CPM_SMATRIX_MAX_ATOMS (two n x n FP64
// work arrays).
int build_sparse_inverse(Ctx* c) {
  const int n = c->n;
  const double* L = c->p.box;
  const bool full = c->p.precond == CPM_PRECOND_FULL;
  const double rc = full ? c->p.rcut_real : c->p.rcut_dc;
  if (n > CPM_SMATRIX_MAX_ATOMS)
    return set_err(c, CPM_EINVAL, "PCG-Normal / PCG-Full: n above CPM_SMATRIX_MAX_ATOMS");
  if (!(rc > 0.0)) return set_err(c, CPM_EINVAL, "PCG-Normal / PCG-Full: cutoff must be positive");
  cudaStream_t s = c->stream;
  Buf& cnt = c->dc_cnt;
  int st;
  if ((st = buf_reserve(c, &cnt, (size_t)n * sizeof(int)))) return st;
  launch_neighbours((const double*)c->xyz.ptr, n, L, rc * rc, (int*)cnt.ptr, nullptr, nullptr,
                    0, full ? 0 : 1, s);
  std::vector<int> hc(n);
  st = cuda_check(c, cudaMemcpyAsync(hc.data(), cnt.ptr, n * sizeof(int),
                                     cudaMemcpyDeviceToHost, s), "pattern counts");
  if (!st) st = cuda_check(c, cudaStreamSynchronize(s), "pattern counts sync");
  if (st) return st;
  std::vector<int64_t> off(n + 1, 0);
  for (int i = 0; i < n; ++i) off[i + 1] = off[i] + hc[i];
  c->nnz = off[n];
  c->pgap = 0.0;
  if ((st = buf_reserve(c, &c->nbr_off, (n + 1) * sizeof(int64_t))) ||
      (st = buf_reserve(c, &c->nbr_idx, c->nnz * sizeof(int))) ||
      (st = buf_reserve(c, &c->prow, c->nnz * sizeof(double))))
    return st;
  st = cuda_check(c, cudaMemcpyAsync(c->nbr_off.ptr, off.data(), (n + 1) * sizeof(int64_t),
                                     cudaMemcpyHostToDevice, s), "pattern offsets");
  if (st) return st;
  launch_neighbours((const double*)c->xyz.ptr, n, L, rc * rc, nullptr,
                    (const int64_t*)c->nbr_off.ptr, (int*)c->nbr_idx.ptr, 1, full ? 0 : 1, s);
  // the columns of E^-1: one PCG over the n identity columns, Jacobi-preconditioned
  Buf ident, cols;
  const size_t bytes = (size_t)n * n * sizeof(double);
  if ((st = buf_alloc(c, &ident, bytes))) return st;
  if ((st = buf_alloc(c, &cols, bytes))) {
    buf_free(c, &ident);
    return st;
  }
  launch_identity((double*)ident.ptr, n, s);
  std::vector<int> it(n);
  std::vector<double> rr(n);
  SolveArgs a{n, (const double*)ident.ptr, 1.0, (double*)cols.ptr, false, 1e-10, 20000,
              it.data(), rr.data()};
  const int saved = c->p.precond;
  c->p.precond = CPM_PRECOND_JACOBI;
  st = pcg_solve(c, a);
  c->p.precond = saved;
  if (!st) {
    (k_gather_inverse<<<n, 128, 0, s>>>(n, (const int64_t*)c->nbr_off.ptr,
                                        (const int*)c->nbr_idx.ptr, (const double*)cols.ptr,
                                        (double*)c->prow.ptr), note_launch());
    st = cuda_check(c, cudaGetLastError(), "gather inverse");
  }
  if (!st) st = cuda_check(c, cudaStreamSynchronize(s), "sparse inverse sync");
  buf_free(c, &ident);
  buf_free(c, &cols);
  return st;
}

__global__ void k_shift(double* __restrict__ v, int64_t len, double s) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len;
       i += (int64_t)gridDim.x * blockDim.x)
    v[i] -= s;
}

// The row form of P on its pattern, as Eq. 36 defines it (the p_gap shift taken back out).
int copy_precond(Ctx* c, int64_t* off, int* idx, double* val) {
  cudaStream_t s = c->stream;
  Buf tmp;
  int st = buf_alloc(c, &tmp, std::max<int64_t>(c->nnz, 1) * sizeof(double));
  if (st) return st;
  st = cuda_check(c, cudaMemcpyAsync(tmp.ptr, c->prow.ptr, c->nnz * sizeof(double),
                                     cudaMemcpyDeviceToDevice, s), "P copy");
  if (!st && c->pgap != 0.0)
    (k_shift<<<256, 256, 0, s>>>((double*)tmp.ptr, c->nnz, -c->pgap), note_launch());
  if (!st) st = cuda_check(c, cudaMemcpyAsync(off, c->nbr_off.ptr, (c->n + 1) * sizeof(int64_t),
                                              cudaMemcpyDefault, s), "P offsets");
  if (!st) st = cuda_check(c, cudaMemcpyAsync(idx, c->nbr_idx.ptr, c->nnz * sizeof(int),
                                              cudaMemcpyDefault, s), "P columns");
  if (!st) st = cuda_check(c, cudaMemcpyAsync(val, tmp.ptr, c->nnz * sizeof(double),
                                              cudaMemcpyDefault, s), "P values");
  if (!st) st = cuda_check(c, cudaStreamSynchronize(s), "P sync");
  buf_free(c, &tmp);
  return st;
}

// p_gap of Eq. 37 from C^ele = 1^T E^-1 1; stored as prow -= p_gap on the pattern.
int apply_p_gap(Ctx* c) {
  double sum_p = 0.0;
  if (int st = device_sum(c, (const double*)c->prow.ptr, c->nnz, &sum_p)) return st;
  const double n2 = (double)c->n * (double)c->n;
  const double nzero = n2 - (double)c->nnz;
  c->pgap = nzero > 0 ? (c->c_ele - sum_p) / nzero : 0.0;
  if (c->pgap != 0.0) (k_shift<<<256, 256, 0, c->stream>>>((double*)c->prow.ptr, c->nnz, c->pgap), note_launch());
  return cuda_check(c, cudaGetLastError(), "p_gap");
}

}  // namespace cpm
