// ortho.cu - FP64 overlap matrices and Gram-Schmidt orthonormalisation of the orbitals.
//
// Orbitals u_{b,k} are cell-normalised: <a|b> = dV sum_r conj(u_a(r)) u_b(r), dV = Omega / N.
// The 4th-order Taylor propagator of Sec. II C is not unitary; the drift of the overlap matrix
// from the identity is the check of a propagation, and orthonormal sets are its input.  Both
// run in FP64 whatever the storage type (complex64 orbitals are widened on load and, for the
// orthonormalisation, rounded once when written back).
//
// Up to 64 bands both run on one Gram kernel: 4 x 4 band tiles per warp, whose 16 products a grid
// point share eight staged values, the points split over a cluster of CTAs that add their sums
// through distributed shared memory in rank order (deterministic, no workspace).  The
// orthonormalisation factorises that matrix per k-point (Cholesky, G = conj(L) L^T) and applies
// L^-1 to the bands point by point: the same vectors as Gram-Schmidt, in two reads and one write
// of the orbitals instead of one sweep per projection.  A k-point whose matrix is not safely well
// conditioned (rounding in L grows with the square of its condition number) is left to the
// modified Gram-Schmidt kernel, which also handles more bands and reports dependent ones.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "launch.cuh"

namespace cg = cooperative_groups;

namespace hse {
namespace {

constexpr int kOrthoThreads = 512;
constexpr int kOverlapThreads = 256;

__device__ __forceinline__ double2 widen(float2 v) { return make_double2(v.x, v.y); }
__device__ __forceinline__ double2 widen(double2 v) { return v; }
__device__ __forceinline__ void narrow(float2* p, double2 v) { *p = make_float2((float)v.x, (float)v.y); }
__device__ __forceinline__ void narrow(double2* p, double2 v) { *p = v; }

// Sum of v over the block (every thread gets it); red: 2 * (blockDim.x / 32) doubles.
__device__ __forceinline__ double2 block_sum2(double2 v, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v.x += __shfl_down_sync(0xffffffffu, v.x, o);
    v.y += __shfl_down_sync(0xffffffffu, v.y, o);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  __syncthreads();  // red is free (a previous sum has been read by every thread)
  if (lane == 0) {
    red[2 * warp] = v.x;
    red[2 * warp + 1] = v.y;
  }
  __syncthreads();
  double2 s = make_double2(0.0, 0.0);
  for (int w = 0; w < nw; ++w) {
    s.x += red[2 * w];
    s.y += red[2 * w + 1];
  }
  return s;
}

// S[k][a][b] = dV sum_r conj(u_a) u_b and S[k][b][a] = conj of it (a real diagonal): block
// (pair a <= b, k); more bands than kGramBands.
template <typename C>
__global__ void __launch_bounds__(kOverlapThreads) overlap_kernel(const C* __restrict__ u, int nb, size_t N, double dV,
                                                                  double2* __restrict__ S) {
  __shared__ double red[2 * (kOverlapThreads / 32)];
  const int k = blockIdx.y;
  int pr = blockIdx.x, a = 0;
  while (pr >= nb - a) {  // pair index -> (a, b) with a <= b, row by row
    pr -= nb - a;
    ++a;
  }
  const int b = a + pr;
  const C* ua = u + ((size_t)k * nb + a) * N;
  const C* ub = u + ((size_t)k * nb + b) * N;
  double2 acc = make_double2(0.0, 0.0);
  for (size_t r = threadIdx.x; r < N; r += blockDim.x) {
    const double2 x = widen(ua[r]), y = widen(ub[r]);
    acc.x = fma(x.x, y.x, fma(x.y, y.y, acc.x));
    acc.y = fma(x.x, y.y, fma(-x.y, y.x, acc.y));
  }
  const double2 s = block_sum2(acc, red);
  if (threadIdx.x == 0) {
    if (a == b) {  // <a|a> is real: its imaginary part is rounding only
      S[((size_t)k * nb + a) * nb + a] = make_double2(dV * s.x, 0.0);
    } else {
      S[((size_t)k * nb + a) * nb + b] = make_double2(dV * s.x, dV * s.y);
      S[((size_t)k * nb + b) * nb + a] = make_double2(dV * s.x, -dV * s.y);
    }
  }
}

constexpr int kGramTiles = 10;   // 4 x 4 band tiles (one warp each) per CTA: all of 16 bands

// One grid point's products of a tile: acc[i][j] += conj(x_i) y_j.  DIAG: j >= i only, and the real
// part on the diagonal.
template <bool DIAG>
__device__ __forceinline__ void gram_point(double2 (&acc)[4][4], const double2 (&x)[4], const double2 (&y)[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int j = DIAG ? i : 0; j < 4; ++j) {
      acc[i][j].x = fma(x[i].x, y[j].x, fma(x[i].y, y[j].y, acc[i][j].x));
      if (!DIAG || i != j) acc[i][j].y = fma(x[i].x, y[j].y, fma(-x[i].y, y[j].x, acc[i][j].y));
    }
  }
}

// S[k][a][b] = dV sum_r conj(u_a) u_b and its Hermitian mirror, nb <= kGramBands.  grid: (cluster of
// CTAs over the points, k, groups of kGramTiles tiles); a warp takes tile warp % kGramTiles' share
// (tiles of this group) and every R-th run of 32 points.
// The FP64 pipe bounds it: 64 multiply-adds a tile and point (32 on the diagonal) against eight
// shared-memory reads; the values are widened once per CTA, when staged.  Two CTAs an SM (96
// registers, a few spills) fill each other's barriers: 64 k x 16 bands at 20^3 989 -> 650 us.
template <typename C>
__global__ void __launch_bounds__(32 * kGramTiles, 2) gram_kernel(const C* __restrict__ u, int nb, size_t N, double dV, double2* __restrict__ S, int tiles_here,
                            int R, const int* __restrict__ skip) {
  extern __shared__ __align__(16) double2 stg[];  // [nbp][32 R]
  __shared__ double red[kGramTiles][33];
  const cg::cluster_group cl = cg::this_cluster();
  const int k = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (skip && skip[k]) return;  // uniform over the cluster
  const int nt = (nb + 3) / 4, ntiles = nt * (nt + 1) / 2, P = 32 * R;
  // 13 to 16 bands: diagonal tiles (0, 4, 7, 9; half the work) go to the schedulers that hold three warps
  // of the ten.  More bands fill several groups of ten, of which only the last can be short; where a
  // group's diagonal tiles lie differs from group to group, and its tiles keep their order.
  constexpr unsigned long long kOrder16 = 0x9786405321ull;
  const int wt = warp % tiles_here, rep = warp / tiles_here;
  const int tl = ntiles == 10 ? (int)((kOrder16 >> (4 * wt)) & 15) : wt;
  const bool on = (int)blockIdx.z * kGramTiles + tl < ntiles;
  int ti = 0, left = on ? blockIdx.z * kGramTiles + tl : 0;
  while (left >= nt - ti) left -= nt - ti++;  // tiles row by row, tj >= ti
  const int tj = ti + left;
  const C* uk = u + (size_t)k * nb * N;
  // this CTA's points, in runs of P
  const size_t runs = (N + P - 1) / P;
  const size_t r0 = cl.block_rank() * runs / cl.num_blocks(), r1 = (cl.block_rank() + 1) * runs / cl.num_blocks();
  double2 acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_double2(0.0, 0.0);
  }
  constexpr int kPre = 8;  // staged elements a thread holds in flight: nbp P <= kPre blockDim
  C pre[kPre];
  auto fetch = [&](size_t run) {
#pragma unroll
    for (int i = 0; i < kPre; ++i) {
      const int e = threadIdx.x + i * blockDim.x, b = e / P;
      const size_t r = run * P + (e - b * P);
      pre[i] = b < nb && r < N ? uk[(size_t)b * N + r] : C{};
    }
  };
  if (r0 < r1) fetch(r0);
  for (size_t run = r0; run < r1; ++run) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kPre; ++i) {
      const int e = threadIdx.x + i * blockDim.x;
      if (e < 4 * nt * P) stg[e] = widen(pre[i]);
    }
    __syncthreads();
    if (run + 1 < r1) fetch(run + 1);
    if (on) {
      double2 x[4], y[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) x[i] = stg[(4 * ti + i) * P + 32 * rep + lane];
      if (ti == tj) {
        gram_point<true>(acc, x, x);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) y[j] = stg[(4 * tj + j) * P + 32 * rep + lane];
        gram_point<false>(acc, x, y);
      }
    }
  }
  // the warp's 32 sums, value v = 8 i + 2 j + part on lane v: each step halves the values a lane
  // carries and adds its partner's
  double v[32];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      v[8 * i + 2 * j] = acc[i][j].x;
      v[8 * i + 2 * j + 1] = acc[i][j].y;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const double mine = up ? v[i + o] : v[i], other = up ? v[i] : v[i + o];
      v[i] = mine + __shfl_xor_sync(0xffffffffu, other, o);
    }
  }
  red[warp][lane] = v[0];
  cl.sync();
  if (cl.block_rank() == 0 && on && rep == 0) {
    double s = 0.0;
    for (int c = 0; c < (int)cl.num_blocks(); ++c) {
      const double* remote = cl.map_shared_rank(&red[0][0], c);
      for (int p = 0; p < R; ++p) s += remote[(p * tiles_here + wt) * 33 + lane];
    }
    s *= dV;
    const int a = 4 * ti + (lane >> 3), b = 4 * tj + ((lane >> 1) & 3), part = lane & 1;
    if (a < nb && b < nb && b >= a) {
      double* Sk = reinterpret_cast<double*>(S + (size_t)k * nb * nb);
      Sk[2 * ((size_t)a * nb + b) + part] = s;
      if (b > a) Sk[2 * ((size_t)b * nb + a) + part] = part ? -s : s;
    }
  }
  cl.sync();  // red stays until rank 0 has read it
}

// Largest bound of the squared condition number (of the matrix scaled to a unit diagonal) at which
// a k-point takes the Cholesky path: rounding in the result is then below 1e-15 x 64 x 1e5 for one
// pass, which complex64 orbitals round away, and a second pass leaves complex128 ones orthonormal
// to rounding.
constexpr double kGramCond2 = 1e5;

// T[k] = L^-1 with S = conj(L) L^T (lower triangular, row-major), one CTA per k-point.  skip[k] = 1
// where S is not positive definite or not safely conditioned (nb sum |T_ab|^2 S_bb > kGramCond2
// bounds the squared condition number of the scaled matrix); k-points already skipped stay so.
__global__ void gram_factor(const double2* __restrict__ S, int nb, double2* __restrict__ T, int* __restrict__ skip,
                            bool first) {
  extern __shared__ __align__(16) double2 lm[];  // L, then T
  double2* tm = lm + nb * nb;
  __shared__ int bad;
  __shared__ double cond;
  const int k = blockIdx.x, tid = threadIdx.x;
  if (!first && skip[k]) return;
  const double2* Sk = S + (size_t)k * nb * nb;
  if (tid == 0) {
    bad = 0;
    cond = 0.0;
  }
  // lm[d][a] (d >= a) starts as S_ad
  for (int i = tid; i < nb * nb; i += blockDim.x) {
    const int d = i / nb, a = i - d * nb;
    lm[i] = d >= a ? Sk[(size_t)a * nb + d] : make_double2(0.0, 0.0);
    tm[i] = make_double2(d == a ? 1.0 : 0.0, 0.0);
  }
  __syncthreads();
  for (int a = 0; a < nb; ++a) {
    const double p = lm[a * nb + a].x;
    const double inv = 1.0 / sqrt(p);
    if (tid == 0 && !(p > 0.0 && p < 1e300)) bad = 1;
    __syncthreads();
    for (int d = a + tid; d < nb; d += blockDim.x)
      lm[d * nb + a] = d == a ? make_double2(p * inv, 0.0) : make_double2(lm[d * nb + a].x * inv, lm[d * nb + a].y * inv);
    for (int b = tid; b <= a; b += blockDim.x) {  // row a of T is final
      tm[a * nb + b].x *= inv;
      tm[a * nb + b].y *= inv;
    }
    __syncthreads();
    // rows f > a: S_ef -= conj(L_ea) L_fa at lm[f][e] for f >= e > a, and T_fe -= L_fa T_ae for e <= a
    const int m = nb - a - 1;
    for (int i = tid; i < m * nb; i += blockDim.x) {
      const int f = a + 1 + i / nb, e = i % nb;
      if (f < e) continue;
      const double2 y = lm[f * nb + a];
      if (e > a) {
        const double2 x = lm[e * nb + a];
        lm[f * nb + e].x -= x.x * y.x + x.y * y.y;
        lm[f * nb + e].y -= x.x * y.y - x.y * y.x;
      } else {
        const double2 x = tm[a * nb + e];
        tm[f * nb + e].x -= x.x * y.x - x.y * y.y;
        tm[f * nb + e].y -= x.x * y.y + x.y * y.x;
      }
    }
    __syncthreads();
  }
  double mine = 0.0;
  for (int i = tid; i < nb * nb; i += blockDim.x) {
    const int b = i % nb;
    mine += (tm[i].x * tm[i].x + tm[i].y * tm[i].y) * Sk[(size_t)b * nb + b].x;
  }
  if (mine != 0.0) atomicAdd(&cond, mine);  // only compared with a bound: the order does not matter
  __syncthreads();
  const bool ok = !bad && nb * cond <= kGramCond2;
  if (tid == 0) skip[k] = ok ? 0 : 1;
  if (!ok) return;
  for (int i = tid; i < nb * nb; i += blockDim.x) T[(size_t)k * nb * nb + i] = tm[i];
}

// u_a <- sum_{b <= a} T_ab u_b in place, one thread a grid point, 16 bands of results at a time
// from the last (so the bands a result reads are still the old ones).  FP64 bound: four
// multiply-adds per element of T, read from shared memory by the whole warp at once.
template <typename C>
__global__ void __launch_bounds__(128) gram_apply(C* __restrict__ u, int nb, size_t N, const double2* __restrict__ T,
                                                  const int* __restrict__ skip) {
  extern __shared__ __align__(16) double2 ts[];  // [16 ceil(nb / 16)][nb]
  const int k = blockIdx.y;
  if (skip[k]) return;
  const int nt = (nb + 15) / 16;
  for (int i = threadIdx.x; i < 16 * nt * nb; i += blockDim.x)
    ts[i] = i < nb * nb ? T[(size_t)k * nb * nb + i] : make_double2(0.0, 0.0);
  __syncthreads();
  const size_t r = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (r >= N) return;
  C* uk = u + (size_t)k * nb * N + r;
  for (int t = nt - 1; t >= 0; --t) {
    double2 acc[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i] = make_double2(0.0, 0.0);
    auto add = [&](int i, int b, double2 w) {
      const double2 c = ts[(16 * t + i) * nb + b];
      acc[i].x = fma(c.x, w.x, fma(-c.y, w.y, acc[i].x));
      acc[i].y = fma(c.x, w.y, fma(c.y, w.x, acc[i].y));
    };
    for (int b = 0; b < 16 * t; ++b) {
      const double2 w = widen(uk[(size_t)b * N]);
#pragma unroll
      for (int i = 0; i < 16; ++i) add(i, b, w);
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      if (16 * t + j >= nb) break;
      const double2 w = widen(uk[(size_t)(16 * t + j) * N]);
#pragma unroll
      for (int i = j; i < 16; ++i) add(i, 16 * t + j, w);
    }
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (16 * t + i < nb) narrow(uk + (size_t)(16 * t + i) * N, acc[i]);
  }
}

// Modified Gram-Schmidt of the nb bands of k-point blockIdx.x, where only[k] is set (every k-point
// where only is null), `passes` times, in w (FP64; for complex64 orbitals a copy, rounded back into
// u at the end; else u itself).  Band a: d = <w_b|w_a> for b = 0, 1, ... a-1 in turn, w_a -= d w_b, then
// w_a /= sqrt(<w_a|w_a>).  Each sweep over the grid applies one projection and accumulates the
// next inner product (with w_{b+1}, or the norm) from the updated values.  A band whose squared
// norm after the projections is at most rel2_min times its squared norm before them (or zero)
// is linearly dependent on the earlier ones: it is set to zero and the status word records
// HSE_ERR_SINGULAR.
template <typename C>
__global__ void __launch_bounds__(kOrthoThreads) gram_schmidt_kernel(C* u, double2* w, int nb, size_t N, double dV,
                                                                      int passes, double rel2_min,
                                                                      const int* __restrict__ only, int* status) {
  __shared__ double red[2 * (kOrthoThreads / 32)];
  if (only && !only[blockIdx.x]) return;
  constexpr bool kCopy = sizeof(C) != sizeof(double2);
  C* uk = u + (size_t)blockIdx.x * nb * N;
  double2* wk = w + (size_t)blockIdx.x * nb * N;
  if constexpr (kCopy) {
    for (size_t r = threadIdx.x; r < nb * N; r += blockDim.x) wk[r] = widen(uk[r]);
    __syncthreads();
  }
  for (int pass = 0; pass < passes; ++pass) {
    for (int a = 0; a < nb; ++a) {
      double2* wa = wk + (size_t)a * N;
      // the norm before the projections, and the first inner product
      double2 n0 = make_double2(0.0, 0.0), d0 = make_double2(0.0, 0.0);
      const double2* w0 = wk;
      for (size_t r = threadIdx.x; r < N; r += blockDim.x) {
        const double2 y = wa[r];
        n0.x = fma(y.x, y.x, fma(y.y, y.y, n0.x));
        if (a > 0) {
          const double2 x = w0[r];
          d0.x = fma(x.x, y.x, fma(x.y, y.y, d0.x));
          d0.y = fma(x.x, y.y, fma(-x.y, y.x, d0.y));
        }
      }
      const double norm0 = block_sum2(n0, red).x * dV;
      double2 d = block_sum2(d0, red);
      d.x *= dV;
      d.y *= dV;
      double norm = norm0;
      for (int b = 0; b < a; ++b) {
        const double2* wb = wk + (size_t)b * N;
        const bool last = b + 1 == a;
        const double2* wn = last ? wa : wk + (size_t)(b + 1) * N;
        double2 acc = make_double2(0.0, 0.0);
        for (size_t r = threadIdx.x; r < N; r += blockDim.x) {
          const double2 x = wb[r];
          double2 y = wa[r];
          y.x -= d.x * x.x - d.y * x.y;
          y.y -= d.x * x.y + d.y * x.x;
          wa[r] = y;
          if (last) {
            acc.x = fma(y.x, y.x, fma(y.y, y.y, acc.x));
          } else {
            const double2 z = wn[r];
            acc.x = fma(z.x, y.x, fma(z.y, y.y, acc.x));
            acc.y = fma(z.x, y.y, fma(-z.y, y.x, acc.y));
          }
        }
        const double2 s = block_sum2(acc, red);
        if (last) {
          norm = s.x * dV;
        } else {
          d = make_double2(s.x * dV, s.y * dV);
        }
      }
      const bool singular = !(norm > rel2_min * norm0) || !(norm0 > 0.0);
      const double scale = singular ? 0.0 : 1.0 / sqrt(norm);
      for (size_t r = threadIdx.x; r < N; r += blockDim.x) {
        const double2 y = wa[r];
        wa[r] = make_double2(y.x * scale, y.y * scale);
      }
      if (singular && threadIdx.x == 0 && status) atomicExch(status, kStatusSingular);
      __syncthreads();  // wa is final before later bands read it
    }
  }
  if constexpr (kCopy) {
    for (size_t r = threadIdx.x; r < nb * N; r += blockDim.x) narrow(uk + r, wk[r]);
  }
}

// S of nb <= kGramBands bands.  The cluster splits the points until the launch has two CTAs an SM.
template <typename C>
cudaError_t launch_gram(const C* u, int nk, int nb, size_t N, double dV, double2* S, const int* skip, cudaStream_t stream) {
  const int nt = (nb + 3) / 4, ntiles = nt * (nt + 1) / 2;
  const int tiles_here = std::min(ntiles, kGramTiles), R = kGramTiles / tiles_here;
  const unsigned groups = (unsigned)((ntiles + kGramTiles - 1) / kGramTiles);
  const size_t runs = (N + 32 * R - 1) / (32 * R);
  unsigned cs = 1;
  while (cs < 8 && (size_t)nk * groups * cs < 2 * 152 && 2 * cs <= runs) cs *= 2;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(cs, (unsigned)nk, groups);
  cfg.blockDim = dim3((unsigned)(32 * tiles_here * R));
  cfg.dynamicSmemBytes = (size_t)4 * nt * 32 * R * sizeof(double2);
  cfg.stream = stream;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = cs;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, gram_kernel<C>, u, nb, N, dV, S, tiles_here, R, skip);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename C>
cudaError_t orthonormalize(C* u, int nk, int nb, size_t N, double dV, double2* work, void* scratch, int* status,
                           cudaStream_t stream) {
  // dependence threshold on the norm ratio: 1e-12 for FP64 data; 1e-5 for complex64, whose
  // rounding leaves about 1e-7 of any band outside the span of the others
  constexpr bool kC128 = sizeof(C) == sizeof(double2);
  const double rel = kC128 ? 1e-12 : 1e-5;
  int* skip = nullptr;
  // The Cholesky path costs four launches (complex128 seven); Gram-Schmidt's sweeps take about
  // 3.4 us (2 + N / 1024) nb (nb + 1) in each wave of k-points (16^3, 8 k, 1 band, complex128: 41
  // against 73 us).
  const double sweeps = 3.4 * nb * (nb + 1.0) * (2.0 + N / 1024.0) * ((nk + 607) / 608);
  if (scratch && sweeps > (kC128 ? 75.0 : 40.0)) {
    double2* S = static_cast<double2*>(scratch);
    double2* T = S + (size_t)nk * nb * nb;
    skip = reinterpret_cast<int*>(T + (size_t)nk * nb * nb);
    const size_t factor_smem = 2 * (size_t)nb * nb * sizeof(double2);
    const size_t apply_smem = (size_t)((nb + 15) / 16 * 16) * nb * sizeof(double2);
    cudaError_t e = cudaSuccess;
    if (factor_smem > 48 * 1024)
      e = cudaFuncSetAttribute(gram_factor, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)factor_smem);
    if (e == cudaSuccess && apply_smem > 48 * 1024)
      e = cudaFuncSetAttribute(gram_apply<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)apply_smem);
    // complex64: one pass (its rounding, below 1e-8 of a band by the conditioning bound, is under that
    // of the result); complex128: twice
    for (int pass = 0; pass < (kC128 ? 2 : 1) && e == cudaSuccess; ++pass) {
      e = launch_gram<C>(u, nk, nb, N, dV, S, pass ? skip : nullptr, stream);
      if (e != cudaSuccess) break;
      gram_factor<<<(unsigned)nk, 128, factor_smem, stream>>>(S, nb, T, skip, pass == 0);
      gram_apply<C><<<dim3((unsigned)((N + 127) / 128), (unsigned)nk), 128, apply_smem, stream>>>(u, nb, N, T, skip);
      count_launch(2);
      e = cudaGetLastError();
    }
    if (e != cudaSuccess) return e;
  }
  gram_schmidt_kernel<C><<<(unsigned)nk, kOrthoThreads, 0, stream>>>(u, work, nb, N, dV, 2, rel * rel, skip, status);
  count_launch();
  return cudaGetLastError();
}

}  // namespace

size_t ortho_scratch_bytes(int nk, int nb) {
  if (nb > kGramBands || nk > 65535) return 0;
  return (size_t)nk * (2 * (size_t)nb * nb * sizeof(double2) + sizeof(int));
}

cudaError_t launch_overlap(bool c128, const void* u, int nk, int nb, size_t N, double dV, double2* S,
                           cudaStream_t stream) {
  if (nb <= kGramBands)
    return c128 ? launch_gram<double2>((const double2*)u, nk, nb, N, dV, S, nullptr, stream)
                : launch_gram<float2>((const float2*)u, nk, nb, N, dV, S, nullptr, stream);
  const dim3 grid((unsigned)(nb * (nb + 1) / 2), (unsigned)nk);
  if (c128)
    overlap_kernel<double2><<<grid, kOverlapThreads, 0, stream>>>((const double2*)u, nb, N, dV, S);
  else
    overlap_kernel<float2><<<grid, kOverlapThreads, 0, stream>>>((const float2*)u, nb, N, dV, S);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_orthonormalize(bool c128, void* u, int nk, int nb, size_t N, double dV, double2* work, void* scratch,
                                  int* status, cudaStream_t stream) {
  return c128 ? orthonormalize<double2>((double2*)u, nk, nb, N, dV, (double2*)u, scratch, status, stream)
              : orthonormalize<float2>((float2*)u, nk, nb, N, dV, work, scratch, status, stream);
}

}  // namespace hse
