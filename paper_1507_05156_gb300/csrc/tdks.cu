// tdks.cu - device pieces of the time propagation around the Fock operator (Sec. II A, II C):
//   * the Taylor-series accumulation of one fourth-order step,
//       term_n = (-i dt / n) (T term_{n-1} + V_x term_{n-1}),  out += term_n;
//   * the spatially averaged electric current (Eqs. current_dns / current_elec without the
//     nonlocal pseudopotential part):  J = -sum_{k,i} (g_s f_{i,k} / N_k) sum_G |c_G|^2 (G+k+A),
//     c_G = (1/N) sum_r u(r) e^{-iG.r}, reduced in FP64 per orbital and then in a fixed order;
//   * the Hartree potential of the orbitals' density (Sec. II A, Eq. tdks-h), FP64:
//       rho(r) = sum_{k,i} (g_s f_{i,k} / N_k) |u_{i,k}(r)|^2,
//       v_H = sum_{G != 0} 4 pi rho~(G) / |G|^2 e^{iG.r}  (G = 0 dropped: neutralising background).
#include <cooperative_groups.h>

#include <algorithm>

#include "fused_f64.cuh"
#include "launch.cuh"

namespace cg = cooperative_groups;

namespace hse {

namespace {

template <typename C>
struct Re;
template <>
struct Re<float2> { using T = float; };
template <>
struct Re<double2> { using T = double; };

// term = (-i s) (kin + vx + vloc prev),  out = base + term;  s = dt / n.  (-i s)(a + ib) = s b - i s a.
// prev: the previous term (may be the same array as term: each element is read, then
// written, by one thread); vloc: [N] real local potential or null; base: psi for the first term,
// then out itself (the same thread reads and writes an element).
template <typename C>
__global__ void taylor_accumulate(const C* __restrict__ kin, const C* __restrict__ vx, const C* prev,
                                  const double* __restrict__ vloc, size_t N, C* term, const C* base, C* out,
                                  size_t count, double s_) {
  using T = typename Re<C>::T;
  const T s = (T)s_;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x) {
    const C a = kin[i], b = vx[i];
    T hx = a.x + b.x, hy = a.y + b.y;
    if (vloc) {
      const T v = (T)vloc[i % N];
      const C p = prev[i];
      hx += v * p.x;
      hy += v * p.y;
    }
    C t;
    t.x = s * hy;
    t.y = -s * hx;
    term[i] = t;
    C o = base[i];
    o.x += t.x;
    o.y += t.y;
    out[i] = o;
  }
}

__device__ __forceinline__ int freq(int i, int n) { return i <= (n - 1) / 2 ? i : i - n; }

// Sum of v over the block's 256 threads, on thread 0; red: 8 doubles.
__device__ __forceinline__ double block_sum(double v, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  for (int w = 0; w < 8; ++w) s += red[w];
  return s;
}

// Moments of orbital blockIdx.x for the current.  With F the unnormalised 3-D transform, Parseval over
// the other two axes gives sum_G |F(G)|^2 m_d = (N / n_d) sum over the pencils of axis d of
// sum_m m |F_d(m)|^2 with the 1-D transform F_d alone, so the three axes (blockIdx.y) are
// independent: one read of the orbital each, no transform is written back, FP64 bound.  partial[o][d]
// gets that sum and (from axis 2) partial[o][3] = sum_r |u|^2.
template <typename C, int LMAX>
__global__ void __launch_bounds__(256) current_moments(const C* __restrict__ u, const CurArgs a, double* __restrict__ partial) {
  __shared__ double red[8];
  const int o = blockIdx.x, d = blockIdx.y;
  const size_t N = (size_t)a.n1 * a.n2 * a.n3;
  const int len = d == 0 ? a.n1 : d == 1 ? a.n2 : a.n3;
  const int stride = d == 0 ? a.n2 * a.n3 : d == 1 ? a.n3 : 1;
  const int pencils = (int)(N / len);
  const C* uo = u + o * N;
  double mom = 0.0, norm = 0.0;
  with_length<LMAX>(len, [&](auto tag) {
    constexpr int L = decltype(tag)::value;
    for (int p = threadIdx.x; p < pencils; p += 256) {
      // axis 0: p = (y, z); axis 1: p = (x, z), planes n2 n3 apart; axis 2: rows
      const size_t base = d == 0 ? p : d == 1 ? (size_t)(p / a.n3) * a.n2 * a.n3 + p % a.n3 : (size_t)p * L;
      cpx<double> v[L];
#pragma unroll
      for (int e = 0; e < L; ++e) {
        const C w = uo[base + (size_t)e * stride];
        v[e] = {(double)w.x, (double)w.y};
      }
      if (d == 2) {
#pragma unroll
        for (int e = 0; e < L; ++e) norm = fma(v[e].x, v[e].x, fma(v[e].y, v[e].y, norm));
      }
      fft<L, -1, double>(v);
#pragma unroll
      for (int e = 1; e < L; ++e) mom += (double)freq(e, L) * fma(v[e].x, v[e].x, v[e].y * v[e].y);
    }
  });
  mom = block_sum(mom, red);
  norm = block_sum(norm, red);
  if (threadIdx.x == 0) {
    partial[4 * (size_t)o + d] = mom / len;
    if (d == 2) partial[4 * (size_t)o + 3] = norm;
  }
}

// J_c = factor * sum_o f_o (sum_d b_d[c] M_d + (k + A)_c |u|^2) (fixed order), factor = -g_s / (N_k N)
__global__ void current_combine(const double* __restrict__ partial, const double* __restrict__ occ, int norb,
                                const CurArgs a, double factor, double* __restrict__ J) {
  __shared__ double red[8];
  double s[3] = {0.0, 0.0, 0.0};
  for (int o = threadIdx.x; o < norb; o += 256) {
    const double* m = partial + 4 * (size_t)o;
    const int k = o / a.nbands;
    for (int c = 0; c < 3; ++c)
      s[c] += occ[o] * (m[0] * a.b[c] + m[1] * a.b[3 + c] + m[2] * a.b[6 + c] + m[3] * (a.kpts[3 * k + c] + a.A[c]));
  }
  for (int c = 0; c < 3; ++c) {
    const double t = block_sum(s[c], red);
    if (threadIdx.x == 0) J[c] = factor * t;
  }
}

// rho[r] = (sum_o w_o |u_o[r]|^2, 0) with w_o = occ[o] * wscale.  A block takes 64 points, four
// threads a point; a cluster of eight splits the orbitals 32 ways and rank 0 adds the shares in
// order (one thread a point looping over every orbital waited for each load: 216 orbitals of 16^3
// took 100 us on 16 SMs).
constexpr int kRhoPoints = 64, kRhoCluster = 8;
template <typename C>
__global__ void __cluster_dims__(kRhoCluster, 1, 1) __launch_bounds__(4 * kRhoPoints)
    hartree_density(const C* __restrict__ u, const double* __restrict__ occ, size_t norb, size_t N, double wscale,
                    double2* __restrict__ rho) {
  __shared__ double part[4][kRhoPoints];
  const cg::cluster_group cl = cg::this_cluster();
  const int p = threadIdx.x % kRhoPoints, g = threadIdx.x / kRhoPoints;
  const size_t r = (size_t)(blockIdx.x / kRhoCluster) * kRhoPoints + p;
  double acc = 0.0;
  if (r < N) {
#pragma unroll 4
    for (size_t o = 4 * cl.block_rank() + g; o < norb; o += 4 * kRhoCluster) {
      const C v = u[o * N + r];
      const double x = (double)v.x, y = (double)v.y;
      acc += occ[o] * (x * x + y * y);
    }
  }
  part[g][p] = acc;
  cl.sync();
  if (cl.block_rank() == 0 && g == 0 && r < N) {
    double s = 0.0;
    for (int c = 0; c < kRhoCluster; ++c) {
      const double* remote = cl.map_shared_rank(&part[0][0], c);
      for (int q = 0; q < 4; ++q) s += remote[q * kRhoPoints + p];
    }
    rho[r] = make_double2(wscale * s, 0.0);
  }
  cl.sync();  // part stays until rank 0 has read it
}

// F(G) <- F(G) 4 pi / (N |G|^2), F(0) <- 0 (F: the unnormalised forward transform of rho)
__global__ void hartree_scale(double2* __restrict__ F, const CurArgs a) {
  const size_t N = (size_t)a.n1 * a.n2 * a.n3;
  for (size_t r = blockIdx.x * (size_t)blockDim.x + threadIdx.x; r < N; r += (size_t)gridDim.x * blockDim.x) {
    const int i3 = (int)(r % a.n3), i2 = (int)((r / a.n3) % a.n2), i1 = (int)(r / ((size_t)a.n3 * a.n2));
    const int m1 = i1 <= (a.n1 - 1) / 2 ? i1 : i1 - a.n1;
    const int m2 = i2 <= (a.n2 - 1) / 2 ? i2 : i2 - a.n2;
    const int m3 = i3 <= (a.n3 - 1) / 2 ? i3 : i3 - a.n3;
    double g2 = 0.0;
    for (int c = 0; c < 3; ++c) {
      const double g = m1 * a.b[c] + m2 * a.b[3 + c] + m3 * a.b[6 + c];
      g2 += g * g;
    }
    const double f = g2 > 0.0 ? 4.0 * 3.14159265358979323846 / ((double)N * g2) : 0.0;
    const double2 v = F[r];
    F[r] = make_double2(v.x * f, v.y * f);
  }
}

__global__ void real_part(const double2* __restrict__ z, double* __restrict__ x, size_t N) {
  for (size_t r = blockIdx.x * (size_t)blockDim.x + threadIdx.x; r < N; r += (size_t)gridDim.x * blockDim.x)
    x[r] = z[r].x;
}

unsigned grid_for(size_t count) { return (unsigned)std::min<size_t>((count + 255) / 256, 152 * 16); }

}  // namespace

cudaError_t launch_taylor_accumulate(bool c128, const void* kin, const void* vx, const void* prev, const double* vloc,
                                     size_t N, void* term, const void* base, void* out, size_t count, double s,
                                     cudaStream_t stream) {
  if (c128)
    taylor_accumulate<double2><<<grid_for(count), 256, 0, stream>>>((const double2*)kin, (const double2*)vx,
                                                                    (const double2*)prev, vloc, N, (double2*)term,
                                                                    (const double2*)base, (double2*)out, count, s);
  else
    taylor_accumulate<float2><<<grid_for(count), 256, 0, stream>>>((const float2*)kin, (const float2*)vx,
                                                                   (const float2*)prev, vloc, N, (float2*)term,
                                                                   (const float2*)base, (float2*)out, count, s);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_current(bool c128, const void* psi, const double* occ, const CurArgs& a, double* partial,
                           double spin_degeneracy, double* J, cudaStream_t stream) {
  const size_t N = (size_t)a.n1 * a.n2 * a.n3;
  const int norb = a.nk * a.nbands;
  const dim3 grid((unsigned)norb, 3);
  const bool small = a.n1 <= 16 && a.n2 <= 16 && a.n3 <= 16;
  if (c128) {
    if (small) current_moments<double2, 16><<<grid, 256, 0, stream>>>((const double2*)psi, a, partial);
    else current_moments<double2, 32><<<grid, 256, 0, stream>>>((const double2*)psi, a, partial);
  } else {
    if (small) current_moments<float2, 16><<<grid, 256, 0, stream>>>((const float2*)psi, a, partial);
    else current_moments<float2, 32><<<grid, 256, 0, stream>>>((const float2*)psi, a, partial);
  }
  current_combine<<<1, 256, 0, stream>>>(partial, occ, norb, a, -spin_degeneracy / ((double)a.nk * (double)N), J);
  count_launch(2);
  return cudaGetLastError();
}

cudaError_t launch_hartree(bool c128, const void* psi, const double* occ, const CurArgs& a, double spin_degeneracy,
                           double2* work, double* vh, cudaStream_t stream) {
  const size_t N = (size_t)a.n1 * a.n2 * a.n3;
  const size_t norb = (size_t)a.nk * a.nbands;
  const double wscale = spin_degeneracy / (double)a.nk;
  const unsigned blocks = (unsigned)((N + kRhoPoints - 1) / kRhoPoints) * kRhoCluster;
  if (c128)
    hartree_density<double2><<<blocks, 4 * kRhoPoints, 0, stream>>>((const double2*)psi, occ, norb, N, wscale, work);
  else
    hartree_density<float2><<<blocks, 4 * kRhoPoints, 0, stream>>>((const float2*)psi, occ, norb, N, wscale, work);
  count_launch();
  cudaError_t e = cudaGetLastError();
  const int inner[3] = {a.n2 * a.n3, a.n3, 1};
  const int len[3] = {a.n1, a.n2, a.n3};
  for (int d = 2; d >= 0 && e == cudaSuccess; --d) e = launch_staged_fft(len[d], -1, work, 1, (int)N, inner[d], stream);
  if (e != cudaSuccess) return e;
  hartree_scale<<<grid_for(N), 256, 0, stream>>>(work, a);
  count_launch();
  e = cudaGetLastError();
  for (int d = 0; d < 3 && e == cudaSuccess; ++d) e = launch_staged_fft(len[d], +1, work, 1, (int)N, inner[d], stream);
  if (e != cudaSuccess) return e;
  real_part<<<grid_for(N), 256, 0, stream>>>(work, vh, N);
  count_launch();
  return cudaGetLastError();
}

}  // namespace hse
