// Host audit of the index arithmetic of the two-CTA pencil-load kernel (8^3, 10^3, 12^3, 18^3, 20^3: one
// pencil a thread, csrc/pairconv_c64.cuh) and of the two-exchange 16^3 kernels (csrc/pairconv_wide.cuh):
// every index stays inside its buffer, the stages cover what they should once, the barriers that
// synchronise less than the CTA guard only what their own threads wrote, and two CTAs fit an SM.  Built
// and run by tests/test_apply_kernels_audit_host.py; exits non-zero on the first violation.
#include <cstdio>
#include <vector>

#include "../../paper_1507_05156_gb300/csrc/launch.cuh"
#include "../../paper_1507_05156_gb300/csrc/pairconv_wide.cuh"

using namespace hse;

static int g_fail = 0;
#define CHECK(cond, ...)              \
  do {                                \
    if (!(cond)) {                    \
      std::printf("FAIL: ");          \
      std::printf(__VA_ARGS__);       \
      std::printf("\n");              \
      ++g_fail;                       \
      return;                         \
    }                                 \
  } while (0)

// Group of thread tid (0-based in the CTA) at the barrier between the Z and Y stages, and the
// threads that the barrier waits for.
template <int n>
static void barrier_group(int tid, int* group, int* count) {
  constexpr int SB = slab_bar_threads<n, 1, Geo<n>::NN>();
  constexpr int threads = GeoP<n, 1, Geo<n>::NN>::THREADS;
  if (SB == 0) {
    *group = 0;
    *count = threads;
  } else if (SB == kSlab20 && n == 20) {
    *group = tid / kSlab20;
    *count = *group == 2 ? 96 : kSlab20;
  } else {
    *group = tid / SB;
    *count = SB;
  }
}

template <int n>
static void audit_two_cta() {
  using G = Geo<n>;
  using GP = GeoP<n, 1, G::NN>;
  CHECK(two_cta_fits(n), "n=%d is not a two-CTA side", n);
  CHECK(2 * GP::TMEM_COLS <= 512 && GP::TMEM_COLS >= 32, "n=%d: TMEM %d columns twice", n, GP::TMEM_COLS);
  CHECK(2 * (pairconv_smem_bytes<n>() + 1024 + 2 * G::NN) <= 233472, "n=%d: shared memory of two CTAs", n);
  CHECK(2 * GP::THREADS <= 2048, "n=%d: %d threads twice", n, GP::THREADS);
  for (int w = 0; w < GP::WARPS; ++w) {
    const int first = (w >> 2) * GP::COLS_PER_WARP;
    CHECK(first + GP::COLS_PER_WARP <= GP::TMEM_COLS, "n=%d: warp %d columns [%d, %d)", n, w, first, first + GP::COLS_PER_WARP);
  }
  CHECK(G::ROW <= GP::TAB && GP::TAB + n <= GP::COLS_PER_WARP, "n=%d: row layout", n);
  constexpr int CH = acc_chunk(n);
  CHECK(CH == 0 || (n % CH == 0 && CH % 2 == 0), "n=%d: chunks of %d", n, CH);
  // barrier groups: whole warps, their sizes add up to the CTA, named barriers 1 to 15
  std::vector<int> members(64, 0), waits(64, 0);
  for (int tid = 0; tid < GP::THREADS; ++tid) {
    int g, c;
    barrier_group<n>(tid, &g, &c);
    ++members[g];
    waits[g] = c;
  }
  constexpr int SB = slab_bar_threads<n, 1, G::NN>();
  for (int g = 0; g < 64; ++g)
    CHECK(members[g] == waits[g] && members[g] % 32 == 0, "n=%d: group %d has %d threads, waits for %d", n, g, members[g], waits[g]);
  for (int g = 15; SB != 32 && g < 64; ++g) CHECK(members[g] == 0, "n=%d: barrier %d", n, 1 + g);
  // the Y stage of a group reads what its own Z stage wrote (thread tid: slot tid / NN, pencil tid % NN)
  std::vector<int> owner((size_t)G::T * G::GRID_CPX, -1), hit((size_t)G::T * G::GRID_CPX, 0);
  for (int tid = 0; tid < G::T * G::NN; ++tid) {
    int g, c;
    barrier_group<n>(tid, &g, &c);
    const int slot = tid / G::NN;
    for (int e = 0; e < n; ++e) {
      const int a = slot * G::GRID_CPX + Pencil<n>(tid % G::NN).zs + e;
      CHECK(a >= 0 && a < G::T * G::GRID_CPX && (size_t)a * 8 < pairconv_smem_bytes<n>(), "n=%d: Z index %d", n, a);
      owner[a] = g;
      ++hit[a];
    }
  }
  int cells = 0;
  for (int h : hit) {
    CHECK(h <= 1, "n=%d: a cell is written twice", n);
    cells += h;
  }
  CHECK(cells == G::T * G::N, "n=%d: %d cells", n, cells);
  for (int tid = 0; tid < G::T * G::NN; ++tid) {
    int g, c;
    barrier_group<n>(tid, &g, &c);
    for (int e = 0; e < n; ++e) {
      const int a = tid / G::NN * G::GRID_CPX + Pencil<n>(tid % G::NN).ys + e * G::P;
      CHECK(a >= 0 && a < G::T * G::GRID_CPX && owner[a] == g, "n=%d: group %d reads a cell of group %d", n, g, owner[a]);
    }
  }
  std::printf("n=%d two CTAs: %d threads, TMEM %d columns, barriers of %d threads closed under Z <-> Y\n", n, GP::THREADS,
              GP::TMEM_COLS, SB ? SB : GP::THREADS);
}

static void audit_wide() {
  using W = Wide16;
  // a slot's grid: what the A stages write is what the B stages read, each cell once
  std::vector<int> a_hit(W::GRID_CPX, 0), cell(W::GRID_CPX, -1);
  for (int t = 0; t < W::TS; ++t)
    for (int k1 = 0; k1 < 4; ++k1)
      for (int z = 0; z < 16; ++z) {
        const WidePlace pl(t);
        const int i = wide_a(pl.hi, pl.lo, 0, 0) + wide_a(0, 0, k1, z);
        CHECK(i >= 0 && i < W::GRID_CPX, "A index %d", i);
        ++a_hit[i];
        cell[i] = ((k1 * 4 + pl.hi) * 16 + pl.lo) * 16 + z;  // (k1, x0, y, z)
      }
  std::vector<int> b_hit(W::GRID_CPX, 0);
  for (int t = 0; t < W::TS; ++t)
    for (int x0 = 0; x0 < 4; ++x0)
      for (int y = 0; y < 16; ++y) {
        const WidePlace pl(t);  // (k1, z)
        const int i = wide_b(pl.hi, pl.lo, 0, 0) + wide_b(0, 0, x0, y);
        CHECK(i >= 0 && i < W::GRID_CPX && cell[i] == ((pl.hi * 4 + x0) * 16 + y) * 16 + pl.lo, "B index %d", i);
        ++b_hit[i];
      }
  int n_a = 0;
  for (int i = 0; i < W::GRID_CPX; ++i) {
    CHECK(a_hit[i] <= 1 && a_hit[i] == b_hit[i], "cell %d: written %d times, read %d times", i, a_hit[i], b_hit[i]);
    n_a += a_hit[i];
  }
  CHECK(n_a == W::N, "%d cells", n_a);
  CHECK(W::SMEM_BYTES == 2u * W::STAGE_BYTES + W::ROW_BYTES + W::SLOTS * W::GRID_CPX * 8u && W::SMEM_REQUEST + 6000 <= 232448,
        "shared memory");
  // half-warps: 16 different 8-byte banks in both stages
  for (int h = 0; h < W::TS; h += 16) {
    int ma = 0, mb = 0;
    for (int l = 0; l < 16; ++l) {
      const WidePlace pl(h + l);
      ma |= 1 << (wide_a(pl.hi, pl.lo, 0, 0) % 16);
      mb |= 1 << (wide_b(pl.hi, pl.lo, 0, 0) % 16);
    }
    CHECK(ma == 0xFFFF && mb == 0xFFFF, "half-warp %d: banks %04x %04x", h / 16, ma, mb);
  }
  // the staged partner: 16-byte chunk e of row p where the 128-byte swizzle puts it, 64 rows on for r
  std::vector<int> s_hit(W::N / 2, 0);
  for (int t = 0; t < W::TS; ++t)
    for (int r = 0; r < 4; ++r)
      for (int e = 0; e < 8; ++e) {
        const WidePlace pl(t);
        const int p0 = pl.hi * 16 + pl.lo, i = wide_stage4(p0, e) + r * 64 * 8, p = (pl.hi + 4 * r) * 16 + pl.lo;
        CHECK(i >= 0 && i < W::N / 2 && i == p * 8 + (e ^ (p % 8)), "stage index %d of row %d", i, p);
        ++s_hit[i];
      }
  for (int h : s_hit) CHECK(h == 1, "a staged chunk is read %d times", h);
  // the kernel row: as stored by the 256 threads, at the place where B thread (k1, z) looks for (k1 + 4 k2, y, z)
  std::vector<int> row(W::N, -1);
  for (int tid = 0; tid < W::THREADS; ++tid) {
    const int t = tid & 63, i0 = tid >> 6;
    const WidePlace pl(t);
    for (int j = 0; j < 4; ++j) {
      const int i = i0 + 4 * j, k2 = i >> 2, y0 = 4 * (i & 3);
      for (int c = 0; c < 4; ++c) {
        const int at = 4 * wide_row4(i, t) + c, v = ((pl.hi + 4 * k2) * 16 + y0 + c) * 16 + pl.lo;
        CHECK(at >= 0 && at < W::N && 4 * at < W::ROW_BYTES && v >= 0 && v < W::N && row[at] < 0, "row index %d", at);
        row[at] = v;
      }
    }
  }
  for (int t = 0; t < W::TS; ++t)
    for (int k2 = 0; k2 < 4; ++k2)
      for (int y = 0; y < 16; ++y) {
        const WidePlace pl(t);
        const int at = 4 * (t + wide_row4(4 * k2 + y / 4, 0)) + y % 4;
        CHECK(row[at] == ((pl.hi + 4 * k2) * 16 + y) * 16 + pl.lo, "row of (%d, %d, %d)", pl.hi + 4 * k2, y, pl.lo);
      }
  // outputs of pfft16: a permutation
  int seen = 0;
  for (int j = 0; j < 16; ++j) seen |= 1 << wide_slot(j);
  CHECK(seen == 0xFFFF, "output slots %04x", seen);
  // running sums (s, then c) and the owner's copy: inside a blocked orbital
  CHECK(31 * W::TS + W::TS - 1 + 32 * W::TS < 2 * (int)(OrbBlk<16>::NBK / 2), "running sums");
  CHECK(31 * W::TS + W::TS - 1 < W::N / 2 && (size_t)W::SLOTS * W::N / 2 <= (size_t)owner_slots(16, kWideVariant) * OrbBlk<16>::NBK / 2,
        "owner copy");
  // Tensor Memory
  for (int w = 0; w < W::WARPS; ++w) CHECK((w >> 2) * W::COLS_PER_WARP + W::OWN + 128 <= 512 && W::ACC + 128 <= W::OWN, "TMEM of warp %d", w);
  std::printf("two-exchange 16^3: %d cells once through each exchange, stage, kernel row, sums and TMEM in bounds\n", n_a);
}

int main() {
  audit_two_cta<8>();
  audit_two_cta<10>();
  audit_two_cta<12>();
  audit_two_cta<18>();
  audit_two_cta<20>();
  audit_wide();
  std::printf(g_fail ? "audit FAILED (%d)\n" : "audit ok\n", g_fail);
  return g_fail ? 1 : 0;
}
