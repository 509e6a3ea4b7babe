// fused_f64.cuh - fused FP64 (complex128) pair-convolution kernel of the Fock-like term.
//
// Same chain as the complex64 kernels (Sec. II C, Eq. "Fock" / "Fock-DS") with the pair's grid in
// shared memory as double2, for any grid whose axes are in the supported set and whose grid fits
// (up to 24^3); the staged form (staged_f64.cuh, one kernel per step through global memory) serves
// the larger ones.  GB300 issues two FP64 multiply-adds a clock and SM, 1/64 of its FP32 rate, so
// the kernel is bound by its FP64 operations, about 59 a grid point and pair at 12^3, and
// everything else only has to stay out of the way: the grid crosses no global memory, orbitals
// and accumulators are read and written once a pair through L2 by the thread that owns the
// z-pencil, and the exchange energy needs no inverse transform at all (Parseval):
//
//   sum_r Re conj(u_i) u_j phi_ji = sum_G v(|G+q|) |F(G)|^2,  F = FFT(conj(u_j) u_i), unnormalised
//
// and, since F_ij(G) = conj(F_ji(-G)), every unordered pair once with v_q(G) + v_-q(-G).
//
// A CTA owns T orbitals (T = 2 where one orbital's pencils would leave the last warp half empty)
// and a range of their partners.  One switch per axis pass selects the register FFT of the axis
// length; an inverse y pass is the forward one on exchanged real and imaginary parts.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fft_reg.cuh"

namespace hse {

enum FusedMode : int {
  F64_APPLY = 0,   // out[k][i] = sum over partners j: owner target, partner occupied
  F64_ENERGY = 1,  // partial[item] = sum over the item's pairs f_i f_j scale sum_G w |F|^2
  F64_OCC = 2,     // VJP w.r.t. the owner (occupied): partners u_i (part) and ybar_i (part2)
};

struct F64Args {
  const double2* own;    // [nk_own][n_own][N]
  const double2* part;   // [nk_part][n_part][N]
  const double2* part2;  // OCC: ybar
  double2* out;          // APPLY / OCC: [nsplit][nk_own][n_own][N]
  double* partial;       // ENERGY: one per item
  const double* occ;     // occupations of the occupied orbitals of the Fock sum [nkq][n_occ]
  const double* occ_own; // ENERGY: [nk_own][n_own]
  const double* vtab;    // [nq][N]
  const int* qidx;       // [target k][sampled k']
  int n1, n2, n3, N;
  int nk_own, nk_part, n_own, n_part, n_occ;
  int ntiles;            // tiles per k-point (ENERGY: tiles of the flattened owners)
  int T, nsplit;
  int stagger;           // items between the CTAs that share an SM (the SM count)
  int mode;
  int sym;               // ENERGY: owners and partners are the same set, unordered pairs once
  double scale;          // -alpha / (N_q N)
};

// most threads of a CTA: two CTAs of 256 threads an SM up to 16 points an axis, one of 512 up to 24
// (128 registers each), one of 256 beyond
constexpr int f64_threads(int longest) { return longest > 16 && longest <= 24 ? 512 : 256; }
constexpr int kF64MaxSmem = 232448 - 1024;  // beside the static part

// pitch of a z-row (odd: neighbouring rows start 16 bytes apart modulo the banks)
__host__ __device__ constexpr int f64_pitch(int n3) { return n3 | 1; }
__host__ __device__ constexpr size_t f64_grid_bytes(int n1, int n2, int n3) {
  return (size_t)n1 * n2 * f64_pitch(n3) * 16;
}

// Threads of a CTA with T orbitals: one a pencil up to f64_threads, and no more than 256 where two
// CTAs' grids fit an SM.
inline int f64_cta_threads(int n1, int n2, int n3, int T) {
  const int longest = n1 > n2 ? (n1 > n3 ? n1 : n3) : (n2 > n3 ? n2 : n3);
  int most = n1 * n2 > n1 * n3 ? n1 * n2 : n1 * n3;
  most = T * (most > n2 * n3 ? most : n2 * n3);
  const int cap = 2 * (T * f64_grid_bytes(n1, n2, n3) + 1024) <= 233472 ? 256 : f64_threads(longest);
  return most < cap ? (most + 31) / 32 * 32 : cap;
}

template <int L>
struct LenTag {
  static constexpr int value = L;
};

// f(LenTag<L>) for the supported axis length n <= LMAX
template <int LMAX, class F>
__device__ __forceinline__ void with_length(int n, F&& f) {
#define HSE_LEN(L)                               \
  case L:                                        \
    if constexpr (L <= LMAX) f(LenTag<L>{});     \
    break;
  switch (n) {
    HSE_LEN(2) HSE_LEN(3) HSE_LEN(4) HSE_LEN(5) HSE_LEN(6) HSE_LEN(8) HSE_LEN(9) HSE_LEN(10) HSE_LEN(12)
    HSE_LEN(15) HSE_LEN(16) HSE_LEN(18) HSE_LEN(20) HSE_LEN(24) HSE_LEN(25) HSE_LEN(27) HSE_LEN(30) HSE_LEN(32)
    default: break;
  }
#undef HSE_LEN
}

// One work item per CTA; grid: nsplit * nk_own * ntiles (ENERGY: nsplit * ntiles), split slowest.
// LMAX: longest axis of the instantiation.
template <int LMAX>
__global__ void __launch_bounds__(f64_threads(LMAX), LMAX <= 12 ? 3 : LMAX <= 16 ? 2 : 1) fused_f64_kernel(const F64Args a) {
  extern __shared__ __align__(16) double2 sm64[];
  __shared__ double red[f64_threads(LMAX) / 32];
  const int tid = threadIdx.x, nt = blockDim.x;
  // pencil of the first round: the CTAs of an SM start one warp apart, so that their last, partial
  // rounds fall on different schedulers (each has its own quarter of the FP64 pipe)
  const int t0 = (tid + 32 * (int)(blockIdx.x / a.stagger)) % nt;
  const int P3 = f64_pitch(a.n3), QS = a.n2 * P3, GS = a.n1 * QS;  // strides of y rows, x planes, slots
  const int n23 = a.n2 * a.n3, n12 = a.n1 * a.n2, n13 = a.n1 * a.n3;
  const bool energy = a.mode == F64_ENERGY, occ_mode = a.mode == F64_OCC;
  const int per_split = energy ? a.ntiles : a.nk_own * a.ntiles;
  const int split = blockIdx.x / per_split, rest = blockIdx.x - split * per_split;
  const int owners = a.nk_own * a.n_own;
  const int k = energy ? 0 : rest / a.ntiles;
  const int o0 = energy ? rest * a.T : k * a.n_own + (rest - k * a.ntiles) * a.T;  // first owner, flattened
  const int T = min(a.T, (energy ? owners : (k + 1) * a.n_own) - o0);
  const long long partners = energy && a.sym ? owners / 2 + 1 : (long long)a.nk_part * a.n_part;
  const int q0 = (int)(split * partners / a.nsplit), q1 = (int)((split + 1) * partners / a.nsplit);
  double2* out = a.out + ((size_t)split * owners + o0) * a.N;
  double esum = 0.0;
  bool first = true;

  for (int q = q0; q < q1; ++q) {
    const int kp = q / a.n_part;
    for (int chain = 0; chain < (occ_mode ? 2 : 1); ++chain) {
      // partner of slot s (flattened index of part)
      auto partner = [&](int s) {
        if (!(energy && a.sym)) return q;
        const int b = o0 + s + q;
        return b < owners ? b : b - owners;
      };
      // pair density conj(x) y, point by point (coalesced; a pass of its own costs a barrier, but the
      // threads that own z-pencils would read the orbitals 16 bytes from 32 lines at a time)
      const double2* prt0 = chain ? a.part2 : a.part;
      for (int i = tid; i < T * a.N; i += nt) {
        const int s = i / a.N, r = i - s * a.N;
        const int row = r / a.n3;
        const double2 o = a.own[(size_t)(o0 + s) * a.N + r], c = prt0[(size_t)partner(s) * a.N + r];
        const double im = o.x * c.y - o.y * c.x;  // of conj(own) partner
        sm64[s * GS + row * P3 + (r - row * a.n3)] = make_double2(o.x * c.x + o.y * c.y, occ_mode ? im : -im);
      }
      __syncthreads();
      // Z, Y, X, and back through Y and Z; an inverse Z or Y pass is the forward one with the parts
      // exchanged, so one set of register FFTs serves all four
#pragma unroll 1
      for (int step = 0; step < (energy ? 3 : 5); ++step) {
        if (step != 2) {
          const bool z_axis = step == 0 || step == 4;
          const int inv = step > 2;
          const int pencils = z_axis ? n12 : n13, stride = 2 * (z_axis ? 1 : P3);
          with_length<LMAX>(z_axis ? a.n3 : a.n2, [&](auto len) {
            constexpr int L = decltype(len)::value;
            for (int p = t0; p < T * pencils; p += nt) {
              const int s = p / pencils, r = p - s * pencils;
              const int x = r / a.n3;  // Y: pencil (x, z)
              double* re = reinterpret_cast<double*>(sm64 + s * GS + (z_axis ? r * P3 : x * QS + (r - x * a.n3))) + inv;
              double* im = re + 1 - 2 * inv;
              cpx<double> v[L];
#pragma unroll
              for (int e = 0; e < L; ++e) v[e] = {re[e * stride], im[e * stride]};
              fft<L, -1, double>(v);
#pragma unroll
              for (int e = 0; e < L; ++e) {
                re[e * stride] = v[e].x;
                im[e * stride] = v[e].y;
              }
            }
          });
          __syncthreads();
          continue;
        }
        // X: forward, kernel multiply, inverse; the energy stops at its weighted square sum
        with_length<LMAX>(a.n1, [&](auto len) {
          constexpr int L = decltype(len)::value;
          for (int p = t0; p < T * n23; p += nt) {
            const int s = p / n23, r = p - s * n23;
            double2* g = sm64 + s * GS + (r / a.n3) * P3 + (r % a.n3);
            cpx<double> v[L];
#pragma unroll
            for (int e = 0; e < L; ++e) {
              const double2 c = g[e * QS];
              v[e] = {c.x, c.y};
            }
            fft<L, -1, double>(v);
            if (energy) {
              const int o = o0 + s, b = partner(s);
              const int ko = o / a.n_own, kb = b / a.n_part;
              const double* w = a.vtab + (size_t)a.qidx[ko * a.nk_part + kb] * a.N + r;
              double sum = 0.0;
              // the ordered term alone: without symmetry, on the diagonal, and at half the circle of
              // an even number of owners, where both ends of the pair come by
              if (!a.sym || q == 0 || 2 * q == owners) {
#pragma unroll
                for (int e = 0; e < L; ++e) sum += w[e * n23] * (v[e].x * v[e].x + v[e].y * v[e].y);
              } else {
                const int y = r / a.n3, z = r - y * a.n3;  // -G
                const double* m = a.vtab + (size_t)a.qidx[kb * a.nk_part + ko] * a.N + (y ? a.n2 - y : 0) * a.n3 +
                                  (z ? a.n3 - z : 0);
#pragma unroll
                for (int e = 0; e < L; ++e)
                  sum += (w[e * n23] + m[(e ? L - e : 0) * n23]) * (v[e].x * v[e].x + v[e].y * v[e].y);
              }
              esum += sum * (a.occ_own[o] * a.occ[b]);
            } else {
              // q = k_i - k_j: APPLY owns i at k, OCC owns j at k
              const int row = occ_mode ? a.qidx[kp * a.nk_own + k] : a.qidx[k * a.nk_part + kp];
              const double* w = a.vtab + (size_t)row * a.N + r;
              const double f = (occ_mode ? a.occ[o0 + s] : a.occ[kp * a.n_occ + (q - kp * a.n_part)]) * a.scale;
#pragma unroll
              for (int e = 0; e < L; ++e) {
                const double wf = w[e * n23] * f;
                v[e].x *= wf;
                v[e].y *= wf;
              }
              fft<L, +1, double>(v);
#pragma unroll
              for (int e = 0; e < L; ++e) g[e * QS] = make_double2(v[e].x, v[e].y);
            }
          }
        });
        __syncthreads();
      }
      if (energy) continue;
      // accumulate: out += w phi (APPLY), w conj(phi) (OCC: the first chain's phi meets ybar, the
      // second's u)
      const double2* w0 = (occ_mode && chain == 0 ? a.part2 : a.part) + (size_t)q * a.N;
      for (int i = tid; i < T * a.N; i += nt) {
        const int s = i / a.N, r = i - s * a.N;
        const int row = r / a.n3;
        double2 v = sm64[s * GS + row * P3 + (r - row * a.n3)];
        if (occ_mode) v.y = -v.y;
        const double2 c = w0[r];
        double2 d = first ? make_double2(0.0, 0.0) : out[i];
        d.x += c.x * v.x - c.y * v.y;
        d.y += c.x * v.y + c.y * v.x;
        out[i] = d;
      }
      first = false;
      __syncthreads();  // the next pair overwrites the grid
    }
  }
  if (!energy) {
    if (first) {  // no partners
      for (int i = tid; i < T * a.N; i += nt) out[i] = make_double2(0.0, 0.0);
    }
    return;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) esum += __shfl_down_sync(0xffffffffu, esum, o);
  if ((tid & 31) == 0) red[tid >> 5] = esum;
  __syncthreads();
  if (tid == 0) {
    double sum = 0.0;
    for (int w = 0; w < nt / 32; ++w) sum += red[w];
    a.partial[blockIdx.x] = sum * a.scale;
  }
}

// Launches the item grid; smem: T grids.
cudaError_t launch_fused_f64(const F64Args& a, cudaStream_t stream);

}  // namespace hse
