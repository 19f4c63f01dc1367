// axis_plan.h -- host-side planning of one FFT axis for the in-place stages of fft_ip.cuh:
// the radices, their order, and the device tables (stages, twiddles, wave numbers).
//
// Used by the library (api.cu) and, compiled for the CPU, by the tests that run the stage
// code on the host.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>
#include <vector>

#include "fft_radix.cuh"   // unit_pair

namespace cbs {

// exp(i a) as a table entry
inline float2 unit_twiddle(double a) {
  const CosSin w = unit_pair(std::cos(a), std::sin(a));
  return make_float2(w.c, w.s);
}

constexpr int kMaxAxisStages = 8;

// How the passes of this axis touch shared memory, for the bank-conflict model.
enum class AxisLayout {
  Rows,      // x passes: elements of a row contiguous; lanes take consecutive butterflies
  Cols,      // y pass: NCOL-column tiles, lanes take column pairs, then butterflies
  ColsZ      // z pass: as Cols, but the last DIF stage moves single columns (the fused
             // k-space stage), lanes taking columns, then butterflies
};

// Factor n into radices of {16, 13, 12, 11, 10, 9, 8, 7, 6, 5, 4, 3, 2} (at most max_radix):
// fewest stages, then the largest smallest radix (fewest threads per transform).  Returns
// false if n has another prime factor.  n = 1 gives the single radix 1.
inline bool factor_radices(int n, int max_radix, std::vector<int>& out) {
  static const int cand[] = {16, 13, 12, 11, 10, 9, 8, 7, 6, 5, 4, 3, 2};
  out.clear();
  if (n == 1) {
    out.push_back(1);
    return true;
  }
  std::vector<int> cur, best;
  auto better = [&](const std::vector<int>& a, const std::vector<int>& b) {
    if (b.empty()) return true;
    if (a.size() != b.size()) return a.size() < b.size();
    return *std::min_element(a.begin(), a.end()) > *std::min_element(b.begin(), b.end());
  };
  std::function<void(int, int)> dfs = [&](int rem, int maxr) {
    if (rem == 1) {
      if (better(cur, best)) best = cur;
      return;
    }
    if ((int)cur.size() >= kMaxAxisStages) return;
    for (int r : cand) {
      if (r > maxr || r > max_radix || rem % r) continue;
      cur.push_back(r);
      dfs(rem / r, r);
      cur.pop_back();
    }
  };
  dfs(n, 1 << 30);
  if (best.empty()) return false;
  out = best;   // largest first
  return true;
}

// Shared-memory wavefronts of one warp-wide access: lane l touches `width` bytes at byte
// address addr[l] (active[l]).  32 banks of 4 bytes; 8-byte accesses are served in two
// phases of 16 lanes, 16-byte ones in four of 8; within a phase the count is the largest
// number of distinct 4-byte words falling in one bank.
inline int warp_wavefronts(const long long* addr, const bool* active, int width) {
  const int per = width >= 16 ? 8 : (width == 8 ? 16 : 32);
  int total = 0;
  for (int ph = 0; ph < 32; ph += per) {
    std::vector<std::vector<long long>> bank(32);
    bool any = false;
    for (int l = ph; l < ph + per; ++l) {
      if (!active[l]) continue;
      any = true;
      for (int w = 0; w < width / 4; ++w) {
        const long long word = addr[l] / 4 + w;
        auto& b = bank[word % 32];
        if (std::find(b.begin(), b.end(), word) == b.end()) b.push_back(word);
      }
    }
    if (!any) continue;
    size_t mx = 0;
    for (auto& b : bank) mx = std::max(mx, b.size());
    total += (int)mx;
  }
  return total;
}

// Modelled shared-memory wavefronts of the element loads of one warp (items 0..31) over all
// stages of `order` (twiddle loads are conflict-free by the table layout), for a tile with
// ncol columns (column layouts) or rows of stride ld (row layout).
inline long long layout_cost(const std::vector<int>& order, int n, AxisLayout lay, int ncol) {
  long long cost = 0;
  int prod = 1;
  const int s = (int)order.size();
  for (int q = 0; q < s; ++q) {
    const int R = order[q];
    prod *= R;
    const int m = n / prod, L = R * m, nb = n / R;
    long long addr[32];
    bool act[32];
    const bool last = (q == s - 1);
    for (int r = 0; r < R; ++r) {
      int width = 8;
      for (int l = 0; l < 32; ++l) {
        act[l] = true;
        if (lay == AxisLayout::Rows) {
          const int t = l % nb;   // items beyond one row wrap to the next row (same banks)
          const int b = t / m, j = t % m;
          if (last && R % 2 == 0) {
            if (r >= R / 2) { act[l] = false; addr[l] = 0; continue; }
            width = 16;
            addr[l] = (long long)(b * L + j) * 8 + 16LL * r;
          } else {
            addr[l] = (long long)(b * L + j + r * m) * 8;
          }
        } else if (lay == AxisLayout::ColsZ && last) {
          const int col = l % ncol, t = (l / ncol) % nb;
          const int b = t / m, j = t % m;
          addr[l] = (long long)((b * L + j + r * m) * ncol + col) * 8;
        } else {
          width = 16;
          const int np = ncol / 2;
          const int p = l % np, t = (l / np) % nb;
          const int b = t / m, j = t % m;
          addr[l] = (long long)((b * L + j + r * m) * np + p) * 16;
        }
      }
      cost += warp_wavefronts(addr, act, width);
    }
  }
  return cost;
}

// The order of the radices for a layout: the permutation with the fewest modelled
// wavefronts; ties keep the largest-first order.
inline std::vector<int> order_radices(const std::vector<int>& radices, int n, AxisLayout lay, int ncol) {
  std::vector<int> perm = radices;
  std::sort(perm.begin(), perm.end());
  std::vector<int> best = radices;
  long long best_cost = layout_cost(radices, n, lay, ncol);
  do {
    const long long c = layout_cost(perm, n, lay, ncol);
    if (c < best_cost) {
      best_cost = c;
      best = perm;
    }
  } while (std::next_permutation(perm.begin(), perm.end()));
  return best;
}

// Modelled work of the stages of one z tile for a radix order: per stage, the rounds a warp
// group of nth threads makes over the stage's items, times the values an item holds.  The
// stages before the last take column pairs of each of the three components (and run twice:
// forward and inverse); the last, fused stage takes single columns with all three
// components and runs its forward and inverse butterflies in one item.  A stage whose items
// leave most threads idle in its last round costs a whole round.
inline long long z_balance_cost(const std::vector<int>& order, int n, int ncol, int nth) {
  long long cost = 0;
  const int s = (int)order.size();
  for (int q = 0; q < s; ++q) {
    const int R = order[q];
    if (q < s - 1) {
      const long long items = 3LL * (ncol / 2) * (n / R);
      cost += 2 * ((items + nth - 1) / nth) * 2 * R;
    } else {
      const long long items = (long long)ncol * (n / R);
      cost += ((items + nth - 1) / nth) * 6 * R;
    }
  }
  return cost;
}

// The order of the z axis' radices: the least modelled work (z_balance_cost), then the fewest
// modelled shared-memory wavefronts (layout_cost), then the largest-first order.
inline std::vector<int> order_radices_z(const std::vector<int>& radices, int n, int ncol, int nth) {
  std::vector<int> perm = radices;
  std::sort(perm.begin(), perm.end());
  std::vector<int> best = radices;
  long long bw = z_balance_cost(radices, n, ncol, nth), bc = layout_cost(radices, n, AxisLayout::ColsZ, ncol);
  do {
    const long long w = z_balance_cost(perm, n, ncol, nth);
    const long long c = layout_cost(perm, n, AxisLayout::ColsZ, ncol);
    if (w < bw || (w == bw && c < bc)) {
      bw = w;
      bc = c;
      best = perm;
    }
  } while (std::next_permutation(perm.begin(), perm.end()));
  return best;
}

// ------------------------------------------------------------- twiddles of the two-step passes
// kTwiddlePhases tables one after the other, `stride` values apart, each used by every
// kTwiddlePhases-th iteration: a value's roundings carry their error on from one table to the
// next, so that over the cycle they average to the value to a fraction of a rounding.  One rounded
// table's errors would act in the same direction in every iteration: they were half of the
// gradient's error (65 x 56 x 48: 2.4 -> 0.7e-6).
constexpr int twiddle_stride(int n) { return (n + 15) / 16 * 16; }

// Twiddles w_n^{j k1} at k1 B + j, j < B = n / A, of every phase.
inline void phased_twiddles(int n, int A, std::vector<float2>& tw) {
  const double two_pi = 6.283185307179586476925287;
  const int B = n / A, stride = twiddle_stride(n);
  tw.assign((size_t)kTwiddlePhases * stride, make_float2(0.f, 0.f));
  for (int k = 0; k < A; ++k)
    for (int j = 0; j < B; ++j) {
      const double a = -two_pi * (double)((long long)j * k % n) / (double)n, c = std::cos(a), s = std::sin(a);
      double cc = 0.0, ss = 0.0;   // carried
      for (int f = 0; f < kTwiddlePhases; ++f) {
        const float2 w = make_float2((float)(c + cc), (float)(s + ss));
        cc += c - (double)w.x;
        ss += s - (double)w.y;
        tw[(size_t)f * stride + k * B + j] = w;
      }
    }
}

// --------------------------------------------------------------- x rows in two steps (xrow.cuh)
// Instructions per value of a radix' in-register transform, roughly: what its split costs (the
// odd primes' symmetric sums, one constant twiddle per value of a split; coprime splits have none,
// but count as the others, as the plans were measured so).
constexpr int radix_cost(int R) {
  if (R <= 2) return R - 1;
  if (R == 4) return 2;
  for (int p : {4, 2, 3, 5, 7, 11, 13})
    if (R % p == 0) return R == p ? p : radix_cost(p) + radix_cost(R / p) + 3;
  return 1 << 20;
}

constexpr bool two_step_radix(int R) {
  return (R >= 2 && R <= 16) || R == 18 || (R >= 20 && R <= 22) || (R >= 24 && R <= 28) || R == 30 || R == 32;
}

constexpr int row_pitch(int B) { return B + (6 - B % 4) % 4; }   // least pitch >= B that is 2 mod 4

// Modelled work of a tile of rpb rows, whole rounds of 32 / B and 32 / A rows counted: step 1
// (radix A) runs both transforms, the update and two twiddle products; step 2 (radix B) runs once
// forward and once inverse, and counts half more from 30 values on, which it moves as 16-byte pairs
// between two warp barriers.  Measured (rows of 64 x 64 grids, us): 400 as 16 x 25 32.7, 20 x 20 37.2,
// 25 x 16 41.1; 275 as 11 x 25 27.2, 25 x 11 30.4; 512 as 16 x 32 39.1, 32 x 16 45.1; 256 as 16 x 16 22.5, 8 x 32
// 22.5, 32 x 8 28.7; 640 x 640 x 336, where memory decides: 32 x 20 2.14 ms, 20 x 32 2.28 ms.
constexpr int row_tile_cost(int A, int B, int rpb) {
  const int per1 = 32 / B, per2 = 32 / A;
  const int w1 = A * (2 * radix_cost(A) + 36), w2 = 2 * B * (radix_cost(B) + 2);
  return (rpb + per1 - 1) / per1 * w1 + (rpb + per2 - 1) / per2 * (B >= 30 ? w2 * 3 / 2 : w2);
}

// The radix A of step 1 of the split n = A B an axis' kernels are built for (0: none): the least
// work per row over tiles of 1, 2 and 4 rows that leave room for six of them (a row of an axis
// too long for that is taken alone).
constexpr int row_split(int n) {
  int at = 0, least = 1 << 30;
  for (int A = 32; A >= 2; --A) {
    const int B = n / A;
    if (A * B != n || !two_step_radix(A) || !two_step_radix(B)) continue;
    for (int rpb = 1; rpb <= 4; rpb *= 2) {
      if (rpb > 1 && 6 * rpb * 8 * (3 * A * row_pitch(B) + 4 * n) > 220 * 1024) continue;
      const int c = row_tile_cost(A, B, rpb) * 4 / rpb;
      if (c < least) {
        least = c;
        at = A;
      }
    }
  }
  return at;
}

// ------------------------------------------------------- columns in two steps (colpass.cuh)
struct ColPlan {
  int A = 0, tx = 0, gt = 0, groups = 0;   // n = A B, columns of a tile, threads of a group, groups
  constexpr int threads() const { return groups * gt + 32; }
};

// Rows of a tensor-copy box of a z tile: the axis in as few boxes as fit (256 rows), each a
// multiple of 128 bytes in shared memory.
constexpr int z_box_rows(int n, int tx) {
  const int nb = (n + 255) / 256, rows = (n + nb - 1) / nb;
  return tx == 8 ? (rows + 1) / 2 * 2 : rows;
}
// Shared memory of a block but its tiles: twiddles, wave numbers (z), mbarriers and flags.
constexpr int col_fixed_smem(int n, int ncomp) {
  return (n + 1) / 2 * 16 * (ncomp == 3 ? 2 : 1) + 8 * 17 + 48;
}
constexpr int kColSmem = 226 * 1024;

// Shape of the y (ncomp = 1) or z (3) kernels of an axis of n; A = 0: none.  Radices up to 32 (z:
// 36 and 12, as step 2 holds three components).  Least modelled time per value: the instructions
// of a group's rounds over a tile's items, at the third of an instruction per cycle that a warp
// issues alone and shared by the groups, plus those of all warps at three per cycle.  Threads
// are kept few enough for the values a thread holds (z of 336 = 28 x 12, 27 million voxels: two
// groups of 288 threads spill at 96 registers, 0.34 ms; of 224, 0.29 ms).  y passes wait for memory,
// so two sets beyond the groups' and tiles of 16 columns count for more there (384: 0.29 against
// 0.31 ms), and so does A < B, whose first step leaves step 2 the shorter rounds (640, forward:
// 20 x 32 1.10 ms, 32 x 20 1.37 ms).
constexpr ColPlan col_plan(int n, int ncomp) {
  ColPlan best;
  double least = 1e300;
  for (int tx = 16; tx >= 8; tx /= 2) {
    if (ncomp == 1 && tx == 8 && n % 2) continue;   // (y boxes must keep 128-byte offsets)
    const int rows = ncomp == 3 ? z_box_rows(n, tx) * ((n + 255) / 256) : n;
    int sets = (kColSmem - col_fixed_smem(n, ncomp)) / (ncomp * rows * tx * 8);
    if (sets > 8) sets = 8;
    if (sets < 3) continue;
    for (int A = 2; A <= 36; ++A) {
      const int B = n / A;
      if (A * B != n || !two_step_radix(B)) continue;
      if (ncomp == 3 ? (B > 12 || !(two_step_radix(A) || A == 35 || A == 36)) : !two_step_radix(A)) continue;
      const int regs = (A > ncomp * B ? A : ncomp * B) * 2;
      const int most = regs > 64 ? 512 : (regs > 50 ? 608 : 736);   // threads: at least 128, 96 or 80 registers
      const double w1 = A * (radix_cost(A) + 8.0) * (ncomp == 3 ? 2 : 1);
      const double w2 = ncomp == 1 ? B * (radix_cost(B) + 3.0) : 6.0 * B * (radix_cost(B) + 2.0) + 34.0 * B;
      const int i1 = ncomp * tx * B, i2 = tx * A;
      for (int gt = 64; gt <= 320; gt += 32) {
        int groups = (most - 32) / gt;
        if (groups > sets - 1) groups = sets - 1;
        if (groups > 6) groups = 6;
        if (groups < 1) continue;
        const double alone = ((i1 + gt - 1) / gt * w1 + (i2 + gt - 1) / gt * w2 + 150.0) * 3.0 / groups;
        const double issue = ((i1 + 31) / 32 * w1 + (i2 + 31) / 32 * w2) / 3.0;
        const double cost = (alone + issue) / (n * tx) * 
                            (ncomp == 1 ? (sets - groups >= 2 ? 1.0 : 1.2) * (tx == 8 ? 1.2 : 1.0) * (A > B ? 1.1 : 1.0) : 1.0);
        if (cost < 0.995 * least) {
          least = cost;
          best.A = A;
          best.tx = tx;
          best.gt = gt;
          best.groups = groups;
        }
      }
    }
  }
  return best;
}

// (p, q) of an axis' table to (p^2, q), the squares from FP64 (a frequency's p is 2 pi k / n).
inline void square_wave_numbers(int n, std::vector<float2>& pq) {
  const double step = 6.283185307179586476925287 / (double)n;
  for (float2& e : pq) {
    const double p = std::round((double)e.x / step) * step;
    e.x = (float)(p * p);
  }
}

// Tables of a column axis: twiddles w_n^{j k1} at k1 B + j; wave numbers by row (y: frequency
// k1 + A k2 sits in row k1 B + (k2 ^ s), s = k1 & 1 for 8 columns and even B) or by frequency (z).
inline void col_tables(int n, const ColPlan& p, bool by_row, std::vector<float2>& tw, std::vector<float2>& pq) {
  const double two_pi = 6.283185307179586476925287;
  const int A = p.A, B = n / A;
  phased_twiddles(n, A, tw);
  pq.assign(n, make_float2(0.f, 0.f));
  for (int k = 0; k < n; ++k) {
    const int k1 = k % A, k2 = k / A, s = (p.tx == 8 && B % 2 == 0) ? k1 & 1 : 0;
    const float q = (float)(two_pi * (double)((2 * k < n) ? k : k - n) / (double)n);
    pq[by_row ? k1 * B + (k2 ^ s) : k] = make_float2(q, (2 * k == n) ? 0.f : q);
  }
}

struct RowPlan {
  int A = 0, B = 0, ldw = 0, lde = 0, rpb = 0, sets = 0, teams = 0;
};

// Tile shape and pitches of an x axis of n with `rows` rows on `sms` processors.  fixed: bytes of
// the tables; budget: shared memory of a block.  A = 0 when the axis has no split.
inline RowPlan plan_rows(int n, long long rows, int sms, size_t budget, size_t fixed) {
  RowPlan best;
  const int A = row_split(n);
  if (!A) return best;
  const int B = n / A, P = row_pitch(B), even = (n + 1) / 2 * 2;
  // pitches free of conflicts between the rows of a round: lanes over j (8-byte accesses), over
  // k1 (16 bytes at pitch P) and over frequencies (8 bytes)
  auto pitch = [&](int least, bool w) {
    int at = least;
    long long lowest = 1LL << 60;
    for (int ld = least; ld < least + 16; ld += 2) {
      long long addr[32], c = 0;
      bool on[32];
      auto fill = [&](int items, int step, int width) {
        for (int l = 0; l < 32; ++l) {
          on[l] = l / items < std::max(1, 32 / items);
          addr[l] = 8LL * ((long long)(l / items) * ld + (long long)(l % items) * step);
        }
        c += warp_wavefronts(addr, on, width);
      };
      fill(B, 1, 8);
      if (w) {
        fill(A, P, 16);
        fill(A, 1, 8);
      }
      if (c < lowest) {
        lowest = c;
        at = ld;
      }
    }
    return at;
  };
  RowPlan p;
  p.A = A;
  p.B = B;
  p.ldw = pitch(std::max(even, A * P), true);
  p.lde = pitch(even, false);
  // rows of a tile and teams: the least work of the busiest processor (its tiles times a tile's
  // work and a tile's fixed part), with a set per team and one in flight unless a single row is
  // too long for that.  Four teams where only they leave room for the better-filled rounds
  // (384 as 24 x 16: two rows 0.665 ms, one row with five teams 0.771 ms; as 16 x 24 0.62), and one
  // team less when the sets just suffice for single rows (640: 2.14 against 2.20 ms).
  double least = 1e300;
  for (int teams : {5, 4})
    for (int rpb = 1; rpb <= 32; ++rpb) {
      const size_t set = (size_t)rpb * (3 * p.ldw + 4 * p.lde) * 8;
      const int sets = (int)std::min<size_t>(8, (budget - fixed) / set);
      if (sets < 2 || (rpb > 1 && sets < teams + 1)) break;
      p.rpb = rpb;
      p.sets = sets;
      p.teams = std::min(rpb == 1 && sets == teams + 1 ? teams - 1 : teams, sets - 1);
      const long long tiles = (rows + rpb - 1) / rpb;
      const double cost = (double)((tiles + sms - 1) / sms) * (row_tile_cost(A, B, rpb) + 50) * (teams == 4 ? 1.03 : 1.0);
      if (cost < 0.99 * least) {
        least = cost;
        best = p;
      }
    }
  return best;
}

// Twiddles w_n^{j k1} at k1 B + j and the wave numbers of the natural order, for plan_rows' axes.
inline void row_tables(int n, const RowPlan& p, std::vector<float2>& tw, std::vector<float2>& pq) {
  const double two_pi = 6.283185307179586476925287;
  phased_twiddles(n, p.A, tw);
  pq.assign(n, make_float2(0.f, 0.f));
  for (int k = 0; k < n; ++k) {
    const float q = (float)(two_pi * (double)((2 * k < n) ? k : k - n) / (double)n);
    pq[k] = make_float2(q, (2 * k == n) ? 0.f : q);
  }
}

// Device tables of an axis for a given radix order (see fft_ip.cuh): the stage table
// (2 int4 per stage), the twiddle table (complex64, w_n^{j k P_q} at tw_off_q + (k-1) m_q + j,
// computed in FP64 and rounded as unit_pair says), and the wave numbers (p, q) of each position (scaled by the
// pitch: p = 2 pi fftfreq(k, n), q = p but 0 at the Nyquist frequency of an even n).
inline void axis_tables(int n, const std::vector<int>& order, std::vector<int4>& st, std::vector<float2>& tw,
                        std::vector<float2>& pq) {
  const double two_pi = 6.283185307179586476925287;
  auto bits = [](float f) {
    int i;
    std::memcpy(&i, &f, sizeof(i));
    return i;
  };
  const int s = (int)order.size();
  st.assign(2 * s, make_int4(1, 1, 1, 0));
  tw.clear();
  int prod = 1;
  for (int q = 0; q < s; ++q) {
    const int R = order[q];
    const int P = prod;   // n / L_q
    prod *= R;
    const int m = n / prod, L = R * m;
    st[2 * q] = make_int4(R, m, L, (int)tw.size());
    st[2 * q + 1] = make_int4(bits(1.0f / (float)m), bits(1.0f / (float)(n / R)), n / R, 0);
    if (q < s - 1)
      for (int k = 1; k < R; ++k)
        for (int j = 0; j < m; ++j) {
          const double a = -two_pi * (double)((long long)j * k * P % n) / (double)n;
          tw.push_back(unit_twiddle(a));
        }
  }
  // position of frequency k: its mixed-radix digits d_q (d_0 least significant, base R_0)
  // weighted by m_q
  pq.assign(n, make_float2(0.f, 0.f));
  for (int k = 0; k < n; ++k) {
    int rem = k, pos = 0, pr = 1;
    for (int q = 0; q < s; ++q) {
      const int R = order[q];
      pr *= R;
      const int d = rem % R;
      rem /= R;
      pos += d * (n / pr);
    }
    const int f = (2 * k < n) ? k : k - n;
    const float p = (float)(two_pi * (double)f / (double)n);
    pq[pos] = make_float2(p, (2 * k == n) ? 0.f : p);
  }
}

}  // namespace cbs
