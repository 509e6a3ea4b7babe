// pairconv_wide.cuh - fused FP32 pair-convolution kernel of the 16^3 grid with two shared-memory
// exchanges per 3-D transform pair instead of four.
//
// Same chain as pairconv_tma.cuh (Sec. II C, Eq. "Fock" / "Fock-DS").  There each thread holds
// one 16-point pencil, so a pair's grid crosses shared memory between every two axes (Z-Y, Y-X,
// X-Y, Y-Z: 64 bytes a grid point).  Here a thread holds 64 points and an owner slot is two
// warps: with x = x0 + 4 r and the X frequency k = k1 + 4 k2,
//
//   A   thread (x0, y): z (16) and r (4):  pair density, FFT along z, the 4-point DFTs over r,
//       twiddles W16^(x0 k1)                                           -> shared memory
//   B   thread (k1, z): y (16) and x0 (4): the 4-point DFTs over x0 (now at k2), FFT along y,
//       multiply by v(|G+q|) * s / N, and back through y and k2 in place -> shared memory
//   A'  thread (x0, y): conjugate twiddles, 4-point DFTs over k1, inverse FFT along z,
//       multiply by the partner and accumulate
//
// so a grid point crosses shared memory twice (32 bytes).  A, B and A' each read and write only
// the thread's own places, so a slot needs two barriers a pair, among its own two warps: the
// four slots of a CTA drift against one another and fill each other's load and barrier gaps.
// What is shared by the slots: the staged partner (two buffers, TMA with the 128-byte swizzle;
// the last of the eight warps to finish with a buffer issues its refill, so nobody waits to
// issue) and the kernel row of the current k' (16 KB, in the order in which the B threads read
// it; swapped under a CTA barrier when k' changes).  TMEM: accumulator and owner orbital, 128
// columns each per warp; the running sums of the compensated accumulation are in global memory
// (PairArgs::comp).  256 threads of up to 255 registers, two warps on every scheduler.
//
// Measured (152 k-points, 16 k', 16 + 16 bands, 622,592 pairs): 8.6 ms staged, 7.18 ms here (3,640
// SM cycles a pair).  FMA pipe 65% busy, issue 58%, shared-memory wavefronts 48%: the two warps of
// a scheduler each keep the pipe busy about 40% of the time when alone and the rest in loads,
// stores, TMEM and barriers, which two independent warps cannot hide completely; registers and
// shared memory leave no room for a third.
#pragma once

#include "pairconv_tma.cuh"

namespace hse {

struct Wide16 {
  static constexpr int n = 16, R = 4, N = 4096;
  static constexpr int SLOTS = 4;                      // owner orbitals per CTA
  static constexpr int TS = 64;                        // threads per slot
  static constexpr int THREADS = SLOTS * TS, WARPS = THREADS / 32;
  // grid of a slot: (x part, y, z) at (4 k1 + x0) Q + y P + z.  A lanes run along y (P = 1 mod
  // 16), B lanes along z: a half-warp's 16 eight-byte accesses always hit 16 different banks.
  static constexpr int P = 17, Q = 272, GRID_CPX = n * Q;
  static constexpr int STAGE_BYTES = N * 8;            // one partner orbital, 128-byte rows
  static constexpr int ROW_BYTES = N * 4;              // one kernel row
  static constexpr size_t SMEM_BYTES = 2 * (size_t)STAGE_BYTES + ROW_BYTES + (size_t)SLOTS * GRID_CPX * 8;
  static constexpr size_t SMEM_REQUEST = SMEM_BYTES + 1024;  // base aligned to 1024 at run time (swizzle)
  static constexpr int ACC = 0, OWN = 128;             // TMEM columns of a warp
  static constexpr int COLS_PER_WARP = 256;
};

// Place of thread t (0..63) of a slot in the A stages: x0 and y; in B: k1 and z.
struct WidePlace {
  int hi, lo;
  __host__ __device__ __forceinline__ explicit WidePlace(int t) : hi(t >> 4), lo(t & 15) {}
};

// Element (k1, z) of the A stages / (x0, y) of B, as smem index of the slot's grid.
__host__ __device__ constexpr int wide_a(int x0, int y, int k1, int z) {
  return (4 * k1 + x0) * Wide16::Q + y * Wide16::P + z;
}
__host__ __device__ constexpr int wide_b(int k1, int z, int x0, int y) {
  return (4 * k1 + x0) * Wide16::Q + y * Wide16::P + z;
}
// 16-byte chunk e (z = 2e, 2e + 1) of staged z-pencil row p = 16 x + y (128-byte TMA swizzle), in float4.
__host__ __device__ constexpr int wide_stage4(int p, int e) { return p * 8 + (e ^ (p & 7)); }
// float4 i = 4 k2 + y / 4 of B thread t in the kernel-row buffer
__host__ __device__ constexpr int wide_row4(int i, int t) { return i * Wide16::TS + t; }

struct WideShared {
  uint64_t mbar[2];
  int done[2];        // warps that have finished with stage buffer b
  int abort;
  float occ[kOccCache];
};

__device__ __forceinline__ void wide_slot_sync(int slot) {
  asm volatile("bar.sync %0, 64;" ::"r"(1 + slot) : "memory");
}

// Complex values in one 64-bit register pair; sums and differences are one packed instruction
// (add / sub.rn.f32x2).  The FP32 pipe is as busy as with scalar ones, but a pair is a quarter
// fewer instructions, and with two warps on a scheduler issue and fetch count: 7.64 -> 7.18 ms
// on 152 k-points, 16 k', 16 + 16 bands.
__device__ __forceinline__ float2 padd(float2 a, float2 b) {
  float2 r;
  asm("add.rn.f32x2 %0, %1, %2;"
      : "=l"(reinterpret_cast<unsigned long long&>(r))
      : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)));
  return r;
}
__device__ __forceinline__ float2 psub(float2 a, float2 b) {
  float2 r;
  asm("sub.rn.f32x2 %0, %1, %2;"
      : "=l"(reinterpret_cast<unsigned long long&>(r))
      : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)));
  return r;
}
// a - i b, a + i b
__device__ __forceinline__ float2 paddmi(float2 a, float2 b) { return make_float2(a.x + b.y, a.y - b.x); }
__device__ __forceinline__ float2 paddpi(float2 a, float2 b) { return make_float2(a.x - b.y, a.y + b.x); }
__device__ __forceinline__ float2 pmul(float2 a, float2 w) {
  return make_float2(a.x * w.x - a.y * w.y, a.x * w.y + a.y * w.x);
}

// Forward 4-point DFT of (a, b, c, d) in place, outputs in order.
__device__ __forceinline__ void pdft4(float2& a, float2& b, float2& c, float2& d) {
  const float2 s0 = padd(a, c), s1 = psub(a, c), t0 = padd(b, d), t1 = psub(b, d);
  a = padd(s0, t0);
  c = psub(s0, t0);
  b = paddmi(s1, t1);
  d = paddpi(s1, t1);
}

// a + c b, a - c b with a real constant c, and a - i c b, a + i c b
__device__ __forceinline__ float2 pfma(float2 a, float c, float2 b) {
  const float2 cc = make_float2(c, c);
  float2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(reinterpret_cast<unsigned long long&>(r))
      : "l"(reinterpret_cast<const unsigned long long&>(cc)), "l"(reinterpret_cast<unsigned long long&>(b)),
        "l"(reinterpret_cast<unsigned long long&>(a)));
  return r;
}
__device__ __forceinline__ float2 pfmami(float2 a, float c, float2 b) {
  return make_float2(fmaf(c, b.y, a.x), fmaf(-c, b.x, a.y));
}

// Last butterfly of a column with twiddles folded in: s0 and s1 are the sum and difference of
// the even inputs, the odd ones are c T0 = c (u1 + u3) and c T1.
__device__ __forceinline__ void pcol(float2& a, float2& b, float2& c_, float2& d, float2 s0, float2 s1, float2 t0,
                                     float2 t1, float c) {
  a = pfma(s0, c, t0);
  c_ = pfma(s0, -c, t0);
  b = pfmami(s1, c, t1);
  d = pfmami(s1, -c, t1);
}

// Forward 16-point DFT in place (4 x 4 Cooley-Tukey).  An inverse transform is this one on
// values with real and imaginary parts exchanged.  Twiddles cost two operations instead of
// four: W = c (1 - i t) is applied as the factor (1 - i t), and the real c, the same for both
// odd inputs of a column, rides on the last butterfly's fused multiply-adds.
__device__ __forceinline__ void pfft16(float2 (&a)[16]) {
  constexpr float c1 = (float)trig2pi(1, 16, 0), h = (float)trig2pi(2, 16, 0);
  constexpr float t = (float)(trig2pi(1, 16, 1) / trig2pi(1, 16, 0));
#pragma unroll
  for (int r = 0; r < 4; ++r) pdft4(a[r], a[4 + r], a[8 + r], a[12 + r]);
  // a[4 k + r] wants the factor exp(-2 pi i r k / 16), then a 4-point DFT over r
  pdft4(a[0], a[1], a[2], a[3]);
  {  // k = 1: W^1 = c1 (1 - i t), W^2 = h (1 - i), W^3 = c1 (t - i)
    const float2 u1 = make_float2(fmaf(t, a[5].y, a[5].x), fmaf(-t, a[5].x, a[5].y));
    const float2 u2 = make_float2(a[6].x + a[6].y, a[6].y - a[6].x);
    const float2 u3 = make_float2(fmaf(t, a[7].x, a[7].y), fmaf(t, a[7].y, -a[7].x));
    pcol(a[4], a[5], a[6], a[7], pfma(a[4], h, u2), pfma(a[4], -h, u2), padd(u1, u3), psub(u1, u3), c1);
  }
  {  // k = 2: W^2 = h (1 - i), W^4 = -i, W^6 = -h (1 + i)
    const float2 u1 = make_float2(a[9].x + a[9].y, a[9].y - a[9].x);
    const float2 u3 = make_float2(a[11].y - a[11].x, -a[11].x - a[11].y);
    pcol(a[8], a[9], a[10], a[11], paddmi(a[8], a[10]), paddpi(a[8], a[10]), padd(u1, u3), psub(u1, u3), h);
  }
  {  // k = 3: W^3 = c1 (t - i), W^6 = -h (1 + i), W^9 = -c1 (1 - i t)
    const float2 u1 = make_float2(fmaf(t, a[13].x, a[13].y), fmaf(t, a[13].y, -a[13].x));
    const float2 u2 = make_float2(a[14].y - a[14].x, -a[14].x - a[14].y);
    const float2 u3 = make_float2(fmaf(t, a[15].y, a[15].x), fmaf(-t, a[15].x, a[15].y));
    pcol(a[12], a[13], a[14], a[15], pfma(a[12], h, u2), pfma(a[12], -h, u2), psub(u1, u3), padd(u1, u3), c1);
  }
}
// Slot of output (or input) j after pfft16: a[4 k + s] holds output k + 4 s.
__host__ __device__ constexpr int wide_slot(int j) { return 4 * (j & 3) + (j >> 2); }

// The 4-point DFTs of v[0..3][e] over the first index, for e = 0..15.
__device__ __forceinline__ void wide_dft4(float2 (&v)[4][16]) {
#pragma unroll
  for (int e = 0; e < 16; ++e) pdft4(v[0][e], v[1][e], v[2][e], v[3][e]);
}

// w[k1 - 1] = exp(-2 pi i x0 k1 / 16)
struct WideTw {
  float2 w[3];
  __device__ __forceinline__ explicit WideTw(int x0) {
#pragma unroll
    for (int k = 1; k < 4; ++k) {
      float s, c;
      sincospif(-0.125f * (float)(x0 * k), &s, &c);
      w[k - 1] = make_float2(c, s);
    }
  }
  __device__ __forceinline__ void apply(float2 (&v)[4][16]) const {
#pragma unroll
    for (int k1 = 1; k1 < 4; ++k1) {
#pragma unroll
      for (int z = 0; z < 16; ++z) v[k1][z] = pmul(v[k1][z], w[k1 - 1]);
    }
  }
};

// One pair chain: `enter` fills v with the pair density, `scale` multiplies by the kernel row and
// exchanges real and imaginary parts (so that the inverse half runs forward transforms),
// `leave` gets phi, parts exchanged, z at wide_slot(z).  Straight-line code (about 60 KB a
// pair): one instance of the transforms in a loop over the four passes fits the instruction
// caches better but keeps loads and stores from overlapping the arithmetic around them and
// spills (9.1 ms against 7.2 ms on 152 k-points, 16 k', 16 + 16 bands).
template <class Enter, class Scale, class Leave>
__device__ __forceinline__ void wide_chain(float2* ga, float2* gb, const WideTw& tw, int slot, Enter&& enter,
                                           Scale&& scale, Leave&& leave) {
  float2 v[4][16];
  // A
  enter(v);
#pragma unroll
  for (int r = 0; r < 4; ++r) pfft16(v[r]);
  wide_dft4(v);
  tw.apply(v);
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) {
#pragma unroll
    for (int z = 0; z < 16; ++z) ga[wide_a(0, 0, k1, z)] = v[k1][wide_slot(z)];
  }
  wide_slot_sync(slot);
  // B
#pragma unroll
  for (int x0 = 0; x0 < 4; ++x0) {
#pragma unroll
    for (int y = 0; y < 16; ++y) v[x0][y] = gb[wide_b(0, 0, x0, y)];
  }
  wide_dft4(v);
#pragma unroll
  for (int k2 = 0; k2 < 4; ++k2) pfft16(v[k2]);
  scale(v);
#pragma unroll
  for (int k2 = 0; k2 < 4; ++k2) pfft16(v[k2]);
  wide_dft4(v);
#pragma unroll
  for (int x0 = 0; x0 < 4; ++x0) {
#pragma unroll
    for (int y = 0; y < 16; ++y) gb[wide_b(0, 0, x0, y)] = v[x0][wide_slot(y)];
  }
  wide_slot_sync(slot);
  // A'
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) {
#pragma unroll
    for (int z = 0; z < 16; ++z) v[k1][z] = ga[wide_a(0, 0, k1, z)];
  }
  tw.apply(v);
  wide_dft4(v);
#pragma unroll
  for (int r = 0; r < 4; ++r) pfft16(v[r]);
  leave(v);
}

// Multiply by the kernel row (row: this thread's float4s) times f and exchange real and
// imaginary parts; y from wide_slot(y) to y.
__device__ __forceinline__ void wide_scale(float2 (&v)[4][16], const float4* row, float f) {
#pragma unroll
  for (int k2 = 0; k2 < 4; ++k2) {
    float2 o[16];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 w = row[wide_row4(4 * k2 + i, 0)];
      const float wf[4] = {w.x * f, w.y * f, w.z * f, w.w * f};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float2 a = v[k2][wide_slot(4 * i + c)];
        o[4 * i + c] = make_float2(a.y * wf[c], a.x * wf[c]);
      }
    }
#pragma unroll
    for (int y = 0; y < 16; ++y) v[k2][y] = o[y];
  }
}

// The owner's four pencils from TMEM (128 columns at town).  Warp-wide.
__device__ __forceinline__ void wide_load_own(float2 (&v)[4][16], uint32_t town) {
#pragma unroll
  for (int r = 0; r < 4; ++r) tmem_issue_row32(town + (uint32_t)(32 * r), reinterpret_cast<float*>(v[r]));
#pragma unroll
  for (int r = 0; r < 4; ++r) tmem_wait_ld32(reinterpret_cast<float*>(v[r]));
}

// v <- conj(a) v with a staged (st); OWN_CONJ: conj(v) a.
template <bool OWN_CONJ>
__device__ __forceinline__ void wide_product(float2 (&v)[4][16], const float4* st, int p0) {
#pragma unroll
  for (int r = 0; r < 4; ++r) {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const float4 w = st[wide_stage4(p0, e) + r * 64 * 8];  // x = x0 + 4 r: 64 rows on
      const float2 a = v[r][2 * e], b = v[r][2 * e + 1];
      const float sg = OWN_CONJ ? -1.f : 1.f;
      v[r][2 * e] = make_float2(w.x * a.x + w.y * a.y, sg * (w.x * a.y - w.y * a.x));
      v[r][2 * e + 1] = make_float2(w.z * b.x + w.w * b.y, sg * (w.z * b.y - w.w * b.x));
    }
  }
}

// Copies one z-pencil set (4 pencils of the thread) of an orbital in the caller's [x][y][z]
// layout into 128 TMEM columns.  Warp-wide.
__device__ __forceinline__ void wide_own_to_tmem(const float2* __restrict__ orb, int x0, int y, uint32_t town) {
#pragma unroll 1
  for (int r = 0; r < 4; ++r) {
    cpx<float> w[16];
    load_pencil_global<16>(w, orb + ((x0 + 4 * r) * 16 + y) * 16);
    float f[32];
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      f[2 * e] = w[e].x;
      f[2 * e + 1] = w[e].y;
    }
    TmemRow<32>::store(town + (uint32_t)(32 * r), f);
  }
}

// acc (TMEM) += epilogue of phi (v, parts exchanged) with the staged orbital st.  Warp-wide.
template <int EPI>
__device__ __forceinline__ void wide_accumulate(const float2 (&v)[4][16], const float4* st, int p0, uint32_t tacc) {
  constexpr int C = 16;  // columns per chunk, the next chunk's load in flight behind each
  float acc[2][C];
  tmem_issue_row16(tacc, acc[0]);
#pragma unroll
  for (int h = 0; h < 128 / C; ++h) {
    float* a = acc[h & 1];
    tmem_wait_ld16(a);
    if (h + 1 < 128 / C) tmem_issue_row16(tacc + (uint32_t)(C * (h + 1)), acc[(h + 1) & 1]);
#pragma unroll
    for (int i = 0; i < C / 4; ++i) {
      const int r = (h * C + 4 * i) / 32, e = (h * C / 4 + i) % 8;
      const float4 w = st[wide_stage4(p0, e) + r * 64 * 8];
      const float2 x = v[r][wide_slot(2 * e)], y = v[r][wide_slot(2 * e + 1)];
      epilogue_mac<EPI>(a[4 * i], a[4 * i + 1], cpx<float>{w.x, w.y}, cpx<float>{x.y, x.x});
      epilogue_mac<EPI>(a[4 * i + 2], a[4 * i + 3], cpx<float>{w.z, w.w}, cpx<float>{y.y, y.x});
    }
    tmem_put_row16(tacc + (uint32_t)(C * h), a);
  }
  tmem_wait_st();
}

// Folds the group sum (TMEM, 128 columns) into the slot's running sums (see fold_group): s in
// sums[0 .. 32) x 64 threads of float4, c behind it.  out: the owner's output orbital, or null
// for an empty slot.  Warp-wide (TMEM).
__device__ __forceinline__ void wide_fold(uint32_t tacc, float4* __restrict__ sums, int t, float2* out, int x0, int y,
                                          bool first, bool second, bool last) {
#pragma unroll 1
  for (int r = 0; r < 4; ++r) {
    float acc[32];
    TmemRow<32>::load(tacc + (uint32_t)(32 * r), acc);
    if (out) {
      float4* s4 = sums + (size_t)(8 * r) * Wide16::TS + t;
      float4* c4 = s4 + 32 * Wide16::TS;
      float4* o4 = reinterpret_cast<float4*>(out + ((x0 + 4 * r) * 16 + y) * 16);
      float4 s0[8], c0[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        s0[e] = first ? make_float4(0.f, 0.f, 0.f, 0.f) : s4[e * Wide16::TS];
        c0[e] = (first || second) ? make_float4(0.f, 0.f, 0.f, 0.f) : c4[e * Wide16::TS];
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        float4 sv = make_float4(acc[4 * e], acc[4 * e + 1], acc[4 * e + 2], acc[4 * e + 3]);
        float4 cv = make_float4(0.f, 0.f, 0.f, 0.f);
        if (!first) fold4(sv, cv, s0[e], c0[e]);
        if (last) {
          o4[e] = make_float4(sv.x + cv.x, sv.y + cv.y, sv.z + cv.z, sv.w + cv.w);
        } else {
          s4[e * Wide16::TS] = sv;
          if (!first) c4[e * Wide16::TS] = cv;
        }
      }
    }
    if (!last) {
#pragma unroll
      for (int e = 0; e < 32; ++e) acc[e] = 0.f;
      TmemRow<32>::store(tacc + (uint32_t)(32 * r), acc);
    }
  }
}

// The kernel row of q (scaled), as 4 float4 of each of the CTA's 256 threads, in the order of
// wide_row4: thread tid holds float4s i = tid / 64 + 4 j of B thread tid % 64.
__device__ __forceinline__ void wide_row_load(float4 (&rv)[4], const float* __restrict__ vrow, float scale) {
  const int t = threadIdx.x & 63, i0 = threadIdx.x >> 6;
  const WidePlace pl(t);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int i = i0 + 4 * j, k2 = i >> 2, y0 = 4 * (i & 3);
    const float* p = vrow + ((pl.hi + 4 * k2) * 16 + y0) * 16 + pl.lo;
    rv[j] = make_float4(__ldg(p) * scale, __ldg(p + 16) * scale, __ldg(p + 32) * scale, __ldg(p + 48) * scale);
  }
}
__device__ __forceinline__ void wide_row_store(const float4 (&rv)[4], float4* row) {
  const int t = threadIdx.x & 63, i0 = threadIdx.x >> 6;
#pragma unroll
  for (int j = 0; j < 4; ++j) row[wide_row4(i0 + 4 * j, t)] = rv[j];
}

// V_x u for a tile of four owners at one k-point over the item's k' range, one item per CTA.
__global__ void __launch_bounds__(Wide16::THREADS, 1)
    pairconv_wide16_kernel(const PairArgs args, const __grid_constant__ CUtensorMap tmap) {
  using W = Wide16;
  extern __shared__ __align__(128) float4 smem4[];
  __shared__ uint32_t tmem_base_sh;
  __shared__ WideShared sh;
  char* sbase = reinterpret_cast<char*>(smem4);
  sbase += (1024u - (smem_addr_u32(sbase) & 1023u)) & 1023u;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int slot = tid / W::TS, t = tid % W::TS;
  const WidePlace pl(t);  // (x0, y) in A, (k1, z) in B
  float2* stage = reinterpret_cast<float2*>(sbase);
  float4* row = reinterpret_cast<float4*>(sbase + 2 * W::STAGE_BYTES);
  float2* g = reinterpret_cast<float2*>(sbase + 2 * W::STAGE_BYTES + W::ROW_BYTES) + slot * W::GRID_CPX;
  if (tid == 0) {
    mbar_init(&sh.mbar[0], 1);
    mbar_init(&sh.mbar[1], 1);
    sh.done[0] = sh.done[1] = 0;
    sh.abort = 0;
    mbar_fence_init();
  }
  if (warp == 0) {
    tmem_alloc(&tmem_base_sh, 512);
    tmem_relinquish();
  }
  const ItemIdx it(args, blockIdx.x);
  const int band = it.tile * W::SLOTS + slot;
  const bool active = band < args.n_own;  // uniform over the slot; an empty slot only passes the CTA barriers
  const int nwarps = 2 * min(W::SLOTS, args.n_own - it.tile * W::SLOTS);  // warps that use the stage
  const int q0 = it.q0, npairs = it.q1 - it.q0, kp_begin = it.q0 / args.n_part;
  for (int i = tid; i < npairs && i < kOccCache; i += W::THREADS) sh.occ[i] = partner_occ(args, q0 + i);
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  const uint32_t tbase = tmem_base_sh;
  const uint32_t tw0 = tbase + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((warp >> 2) * W::COLS_PER_WARP);
  const uint32_t tacc = tw0 + W::ACC, town = tw0 + W::OWN;

  // fill stage buffer `buf` with partner q (one thread)
  auto fill = [&](int q, int buf) {
    mbar_arrive_expect_tx(&sh.mbar[buf], (uint32_t)W::STAGE_BYTES);
    tensor_copy_2d_g2s(stage + buf * W::N, &tmap, 0, (q0 + q) * 256, &sh.mbar[buf]);
  };
  int q = next_partner(sh.occ, args, q0, 0, npairs);
  int q1 = q < npairs ? next_partner(sh.occ, args, q0, q + 1, npairs) : npairs;
  if (tid == 0 && args.inject != 1) {
    if (q < npairs) fill(q, 0);
    if (q1 < npairs) fill(q1, 1);
  }

  // owner orbital into TMEM, accumulators to zero
  const size_t oofs = it.split * args.split_stride + ((size_t)it.k * args.n_own + (active ? band : 0)) * W::N;
  float4* sums = sums_of(args, oofs / W::N, OrbBlk<16>::NBK);
  float2* out = active ? args.out + oofs : nullptr;
  if (active) {
    wide_own_to_tmem(args.own + ((size_t)it.k * args.n_own + band) * W::N, pl.hi, pl.lo, town);
    float z[32];
#pragma unroll
    for (int e = 0; e < 32; ++e) z[e] = 0.f;
#pragma unroll
    for (int r = 0; r < 4; ++r) TmemRow<32>::store(tacc + (uint32_t)(32 * r), z);
  }
  const WideTw tw(pl.hi);
  float2* ga = g + wide_a(pl.hi, pl.lo, 0, 0);
  float2* gb = g + wide_b(pl.hi, pl.lo, 0, 0);
  const int p0 = pl.hi * 16 + pl.lo;  // staged row of r = 0
  const int fspan = fold_terms(args.n_part, args.nk_part) / args.n_part;
  int folds = 0;
  uint32_t phases = 0;  // bit b: parity that stage buffer b completes next
  int buf = 0, cur_kp = -1;
  while (q < npairs) {
    const int kp = (q0 + q) / args.n_part;
    const float f = item_occ(sh.occ, args, q0, q);
    if (kp != cur_kp) {  // uniform over the CTA
      float4 rv[4];
      wide_row_load(rv, args.vtab + (size_t)args.qidx[it.k * args.nk_part + kp] * W::N, args.scale);
      if (active && cur_kp >= 0 && (kp - kp_begin) / fspan != (cur_kp - kp_begin) / fspan) {
        wide_fold(tacc, sums, t, out, pl.hi, pl.lo, folds == 0, folds == 1, false);
        ++folds;
      }
      __syncthreads();  // every slot is past its last use of the old row
      wide_row_store(rv, row);
      __syncthreads();
      cur_kp = kp;
    }
    const int q2 = q1 < npairs ? next_partner(sh.occ, args, q0, q1 + 1, npairs) : npairs;
    if (active) {
      if (!sh.abort && !mbar_wait_bounded(&sh.mbar[buf], (phases >> buf) & 1u)) {
        sh.abort = 1;
        if (args.status) atomicExch(args.status, kStatusTimeout);
      }
      const float4* st = reinterpret_cast<const float4*>(stage + buf * W::N);
      wide_chain(
          ga, gb, tw, slot, [&](float2 (&v)[4][16]) {
            wide_load_own(v, town);
            wide_product<false>(v, st, p0);
          },
          [&](float2 (&v)[4][16]) { wide_scale(v, row + t, f); },
          [&](float2 (&v)[4][16]) { wide_accumulate<EPI_MUL>(v, st, p0, tacc); });
      // the last warp to finish with this buffer refills it with the partner after next (a
      // warp cannot come back to the buffer before that refill has landed)
      __syncwarp();
      if (lane == 0) {
        __threadfence_block();
        if (atomicAdd(&sh.done[buf], 1) == nwarps - 1) {
          sh.done[buf] = 0;
          __threadfence_block();
          if (q2 < npairs && !sh.abort) {
            fence_proxy_async_smem();
            fill(q2, buf);
          }
        }
      }
    }
    phases ^= 1u << buf;
    q = q1;
    q1 = q2;
    buf ^= 1;
  }
  __syncthreads();
  if (tid == 0 && sh.abort) {
    // a copy may still be in flight after a timeout: give it one more bounded chance to land
    mbar_wait_bounded(&sh.mbar[0], phases & 1u);
    mbar_wait_bounded(&sh.mbar[1], (phases >> 1) & 1u);
  }
  if (active) wide_fold(tacc, sums, t, out, pl.hi, pl.lo, folds == 0, folds == 1, true);
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  if (warp == 0) tmem_dealloc(tbase, 512);
}

// The VJP with respect to the occupied orbitals (MODE_OCC) for a tile of four owners u_j at one k':
// per partner (u_i, ybar_i) the two chains phi = K(conj(u_j) u_i), acc += conj(phi) ybar_i and
// psi = K(conj(u_j) ybar_i), acc += u_i conj(psi), which differ only in which of the two staged
// arrays is the factor and which is met at the end.  One stage buffer each: the pairs alternate
// which chain comes first, so the array that the next pair's first chain starts from is the one
// this pair has been done with since the start of its second chain, and the other one lands while
// that first chain is under way.
//
// FUSE_W: the omega gradient rides on the transforms (args.vtab2): the first chain keeps its
// spectrum A and the second adds Re sum_G dv A conj(B), as stage_x_occ does.  A takes the owner's
// TMEM columns and the owner comes from a copy in the order of the threads (args.spec, one blocked
// grid a slot), which 32 loads fetch at the start of a chain, when the registers are free for all of
// them.  Of the 299 us omega costs, those loads are 136, the loads of dv 50, the FP64 sums of 16 products each 46
// (A in that scratch and the owner in TMEM: 40 more, its loads a few at a time between live spectra).
// 16^3, 3^3 k, 8 bands: 1,546 us on the pencil-load kernel with omega, 1,429 here; 1,387 and 1,130 us
// without.
template <bool FUSE_W>
__global__ void __launch_bounds__(Wide16::THREADS, 1)
    pairconv_wide16_occ_kernel(const PairArgs args, const __grid_constant__ CUtensorMap tmap_u,
                               const __grid_constant__ CUtensorMap tmap_y) {
  using W = Wide16;
  extern __shared__ __align__(128) float4 smem4[];
  __shared__ uint32_t tmem_base_sh;
  __shared__ uint64_t mbar[2];
  __shared__ int done[2], fills[2], abort_sh;
  __shared__ double red[FUSE_W ? W::THREADS : 1];
  char* sbase = reinterpret_cast<char*>(smem4);
  sbase += (1024u - (smem_addr_u32(sbase) & 1023u)) & 1023u;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int slot = tid / W::TS, t = tid % W::TS;
  const WidePlace pl(t);
  float2* stage = reinterpret_cast<float2*>(sbase);  // [0] u_i, [1] ybar_i
  float4* row = reinterpret_cast<float4*>(sbase + 2 * W::STAGE_BYTES);
  float2* g = reinterpret_cast<float2*>(sbase + 2 * W::STAGE_BYTES + W::ROW_BYTES) + slot * W::GRID_CPX;
  if (tid == 0) {
    mbar_init(&mbar[0], 1);
    mbar_init(&mbar[1], 1);
    done[0] = done[1] = fills[0] = fills[1] = 0;
    abort_sh = 0;
    mbar_fence_init();
  }
  if (warp == 0) {
    tmem_alloc(&tmem_base_sh, 512);
    tmem_relinquish();
  }
  const int item = args.item0 + blockIdx.x;
  const ItemIdx it(args, item);
  const int band = it.tile * W::SLOTS + slot;
  const bool active = band < args.n_own;  // uniform over the slot
  const int nwarps = 2 * min(W::SLOTS, args.n_own - it.tile * W::SLOTS);
  const int npairs = it.q1 - it.q0, kp_begin = it.q0 / args.n_part;
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  const uint32_t tbase = tmem_base_sh;
  const uint32_t tw0 = tbase + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((warp >> 2) * W::COLS_PER_WARP);
  const uint32_t tacc = tw0 + W::ACC, town = tw0 + W::OWN;
  auto fill = [&](int q, int b) {  // one thread
    ++fills[b];
    mbar_arrive_expect_tx(&mbar[b], (uint32_t)W::STAGE_BYTES);
    tensor_copy_2d_g2s(stage + b * W::N, b ? &tmap_y : &tmap_u, 0, (it.q0 + q) * 256, &mbar[b]);
  };
  if (tid == 0 && args.inject != 1 && npairs > 0) {
    fill(0, 0);
    fill(0, 1);
  }
  const size_t oofs = it.split * args.split_stride + ((size_t)it.k * args.n_own + (active ? band : 0)) * W::N;
  float4* sums = sums_of(args, oofs / W::N, OrbBlk<16>::NBK);
  float2* out = active ? args.out + oofs : nullptr;
  // FUSE_W: this thread's 32 float4 of the owner, 64 float4 apart
  float4* own4 = FUSE_W ? reinterpret_cast<float4*>(args.spec) + ((size_t)blockIdx.x * W::SLOTS + slot) * (W::N / 2) + t : nullptr;
  if (active) {
    const float2* own = args.own + ((size_t)it.k * args.n_own + band) * W::N;
    if constexpr (FUSE_W) {
#pragma unroll 8
      for (int i = 0; i < 32; ++i)
        own4[i * W::TS] = __ldg(reinterpret_cast<const float4*>(own + ((pl.hi + 4 * (i >> 3)) * 16 + pl.lo) * 16) + (i & 7));
    } else {
      wide_own_to_tmem(own, pl.hi, pl.lo, town);
    }
    float z[32];
#pragma unroll
    for (int e = 0; e < 32; ++e) z[e] = 0.f;
#pragma unroll
    for (int r = 0; r < 4; ++r) TmemRow<32>::store(tacc + (uint32_t)(32 * r), z);
  }
  const WideTw tw(pl.hi);
  float2* ga = g + wide_a(pl.hi, pl.lo, 0, 0);
  float2* gb = g + wide_b(pl.hi, pl.lo, 0, 0);
  const int p0 = pl.hi * 16 + pl.lo;
  const float f = active ? (float)args.occ[it.k * args.n_occ + band] : 0.f;
  double wsum = 0.0;
  const int fspan = fold_terms(args.n_part, args.nk_part) / args.n_part;
  int folds = 0, cur_kp = -1;
  const float* dv0 = nullptr;
  for (int q = 0; q < npairs; ++q) {
    const int kp = (it.q0 + q) / args.n_part;
    if (kp != cur_kp) {  // uniform over the CTA
      const size_t qrow = args.qidx[kp * args.nk_own + it.k];
      float4 rv[4];
      wide_row_load(rv, args.vtab + qrow * W::N, args.scale);
      if (active && cur_kp >= 0 && (kp - kp_begin) / fspan != (cur_kp - kp_begin) / fspan) {
        wide_fold(tacc, sums, t, out, pl.hi, pl.lo, folds == 0, folds == 1, false);
        ++folds;
      }
      __syncthreads();  // every slot is past its last use of the old row
      wide_row_store(rv, row);
      __syncthreads();
      cur_kp = kp;
      if (FUSE_W) dv0 = args.vtab2 + qrow * W::N + pl.hi * 256 + pl.lo;  // element (x = k1 + 4 k2, y, z) at (4 k2 16 + y) 16
    }
    if (!active) continue;
    auto wait = [&](int b) {
      if (!abort_sh && !mbar_wait_bounded(&mbar[b], (uint32_t)q & 1u)) {
        abort_sh = 1;
        if (args.status) atomicExch(args.status, kStatusTimeout);
      }
    };
    // the last warp to finish with buffer b refills it with the next partner's array
    auto release = [&](int b) {
      __syncwarp();
      if (lane == 0) {
        __threadfence_block();
        if (atomicAdd(&done[b], 1) == nwarps - 1) {
          done[b] = 0;
          __threadfence_block();
          if (q + 1 < npairs && !abort_sh) {
            fence_proxy_async_smem();
            fill(q + 1, b);
          }
        }
      }
    };
#pragma unroll 1
    for (int c = 0; c < 2; ++c) {
      const int b = (q + c) & 1;  // factor; b ^ 1 is met at the end
      const float4* sp = reinterpret_cast<const float4*>(stage + b * W::N);
      const float4* se = reinterpret_cast<const float4*>(stage + (b ^ 1) * W::N);
      if (c == 0) wait(b);
      wide_chain(
          ga, gb, tw, slot,
          [&](float2 (&v)[4][16]) {
            if constexpr (FUSE_W) {
#pragma unroll
              for (int i = 0; i < 32; ++i) {
                const float4 o = own4[i * W::TS];
                v[i >> 3][2 * (i & 7)] = make_float2(o.x, o.y);
                v[i >> 3][2 * (i & 7) + 1] = make_float2(o.z, o.w);
              }
            } else {
              wide_load_own(v, town);
            }
            wide_product<true>(v, sp, p0);
            if (c == 1) release(b);
          },
          [&](float2 (&v)[4][16]) {
            if (FUSE_W && c == 0) {
#pragma unroll
              for (int k2 = 0; k2 < 4; ++k2) tmem_put_row32(town + (uint32_t)(32 * k2), reinterpret_cast<const float*>(v[k2]));
              tmem_wait_st();
            } else if (FUSE_W) {
#pragma unroll
              for (int k2 = 0; k2 < 4; ++k2) {
                float d = 0.f;
                float2 a[16];
                tmem_issue_row32(town + (uint32_t)(32 * k2), reinterpret_cast<float*>(a));
                float w[16];
#pragma unroll
                for (int y = 0; y < 16; ++y) w[y] = __ldg(dv0 + k2 * 1024 + y * 16);
                tmem_wait_ld32(reinterpret_cast<float*>(a));
#pragma unroll
                for (int y = 0; y < 16; ++y) {
                  const int i = wide_slot(y);
                  d = fmaf(w[y], fmaf(a[i].x, v[k2][i].x, a[i].y * v[k2][i].y), d);
                }
                wsum += (double)d;  // 16 products to an FP32 sum, as in the pencil kernels
              }
            }
            wide_scale(v, row + t, f);
          },
          [&](float2 (&v)[4][16]) {
            if (c == 0) wait(b ^ 1);
            wide_accumulate<EPI_CONJPHI>(v, se, p0, tacc);
            if (c == 1) release(b ^ 1);
          });
    }
  }
  __syncthreads();
  if (tid == 0 && abort_sh) {
    // a copy may still be in flight after a timeout: give it one more bounded chance to land
    for (int b = 0; b < 2; ++b)
      if (fills[b] > 0) mbar_wait_bounded(&mbar[b], (uint32_t)(fills[b] - 1) & 1u);
  }
  if (active) wide_fold(tacc, sums, t, out, pl.hi, pl.lo, folds == 0, folds == 1, true);
  if constexpr (FUSE_W) {  // the item's share of d/d omega, one FP64 partial
    red[tid] = active ? wsum * (double)(args.scale * f) : 0.0;
    __syncthreads();
    if (tid == 0) {
      double sum = 0.0;
      for (int e = 0; e < W::THREADS; ++e) sum += red[e];
      args.partial2[item] = sum;
    }
  }
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  if (warp == 0) tmem_dealloc(tbase, 512);
}

}  // namespace hse
