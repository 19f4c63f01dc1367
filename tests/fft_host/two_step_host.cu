// two_step_host.cu -- the two-step transforms of the CUDA library (axis_plan.h, fft_radix.cuh) on the
// CPU for the tests: the codelets, the phased twiddle tables, the axis plans, and both steps with the
// positions that xrow.cuh and colpass.cuh use.  Built for the host only; not part of the library.
#include <vector>

#include "axis_plan.h"
#include "fft_radix.cuh"

using namespace cbs;

namespace {

template <bool INV, int... R>
bool run_dft(int r, float2* v, std::integer_sequence<int, R...>) {
  bool done = false;
  auto one = [&](auto ri) {
    constexpr int N = decltype(ri)::value;
    if constexpr (N >= 2 && (two_step_radix(N) || N == 35 || N == 36))
      if (r == N) {
        DFT<N, INV>::run(v);
        done = true;
      }
  };
  (one(std::integral_constant<int, R>{}), ...);
  return done;
}
bool dft(int r, bool inv, float2* v) {
  const auto all = std::make_integer_sequence<int, 37>{};
  return inv ? run_dft<true>(r, v, all) : run_dft<false>(r, v, all);
}
float2 conj(float2 a) { return make_float2(a.x, -a.y); }

// Row (or position) of value (k1, j) or (k1, k2) between and after the steps of a column tile.
int col_row(const ColPlan& p, int B, int k1, int j) { return k1 * B + (j ^ (p.tx == 8 && B % 2 == 0 ? k1 & 1 : 0)); }

}  // namespace

extern "C" {

int ts_dft(int r, int inv, float* v) { return dft(r, inv != 0, reinterpret_cast<float2*>(v)) ? 0 : -1; }

// which: 0 x, 1 y, 2 z.  out: A, then (y, z) columns, threads of a group, groups, sets, rows held a
// component, rows of a box; (x) pitches of W and of E and V, rows of a tile, sets, teams.
int ts_plan(int n, int which, long long rows, int* out) {
  if (which == 0) {
    const RowPlan p = plan_rows(n, rows, 152, 226 * 1024, (size_t)(n + 1) / 2 * 16 + 8 * 17 + 16);
    const int v[6] = {p.A, p.ldw, p.lde, p.rpb, p.sets, p.teams};
    for (int i = 0; i < 6; ++i) out[i] = v[i];
    return 6;
  }
  const ColPlan p = col_plan(n, which == 1 ? 1 : 3);
  const int box = which == 1 ? n : z_box_rows(n, p.tx), held = which == 1 ? n : box * ((n + 255) / 256);
  const int ncomp = which == 1 ? 1 : 3;
  const int sets = p.A ? (kColSmem - col_fixed_smem(n, ncomp)) / (ncomp * held * p.tx * 8) : 0;
  const int v[7] = {p.A, p.tx, p.gt, p.groups, sets > 8 ? 8 : sets, held, box};
  for (int i = 0; i < 7; ++i) out[i] = v[i];
  return 7;
}

// The twiddles of a phase, k1 B + j.
void ts_twiddles(int n, int A, int phase, float* out) {
  std::vector<float2> tw;
  phased_twiddles(n, A, tw);
  std::memcpy(out, &tw[(size_t)phase * twiddle_stride(n)], n * sizeof(float2));
}

// A column (which 1, 2) or row (0) of n values through both steps at `phase`: forward leaves the
// spectrum where the kernels do (out[i]: the value in row i; freq[i]: the frequency its table names);
// inverse undoes it.
int ts_transform(int n, int which, int phase, int inv, const float* in, float* out, int* freq) {
  const ColPlan p = which ? col_plan(n, which == 1 ? 1 : 3) : ColPlan{};
  const int A = which ? p.A : row_split(n);
  if (!A) return -1;
  const int B = n / A;
  std::vector<float2> tw, pq;
  if (which == 0) {
    RowPlan r;
    r.A = A;
    r.B = B;
    row_tables(n, r, tw, pq);
  } else {
    col_tables(n, p, which == 1, tw, pq);
  }
  const float2* const w = &tw[(size_t)phase * twiddle_stride(n)];
  // the memory position of frequency k1 + A k2: its row (y), or the frequency itself (x; z, on chip)
  auto place = [&](int k1, int k2) { return which == 1 ? col_row(p, B, k1, k2) : k1 + A * k2; };
  auto between = [&](int k1, int j) { return which ? col_row(p, B, k1, j) : k1 * B + j; };
  const float2* const x = reinterpret_cast<const float2*>(in);
  float2* const y = reinterpret_cast<float2*>(out);
  std::vector<float2> mid(n);
  float2 v[40];
  for (int i = 0; i < n; ++i) {   // (p, q): p = 2 pi k / n
    const int k = (int)std::lround((double)pq[i].x * n / 6.283185307179586);
    freq[i] = (k + n) % n;
  }
  if (!inv) {
    for (int j = 0; j < B; ++j) {
      for (int r = 0; r < A; ++r) v[r] = x[j + B * r];
      if (!dft(A, false, v)) return -1;
      for (int k1 = 0; k1 < A; ++k1) mid[between(k1, j)] = k1 ? cmul(v[k1], w[k1 * B + j]) : v[0];
    }
    for (int k1 = 0; k1 < A; ++k1) {
      for (int j = 0; j < B; ++j) v[j] = mid[between(k1, j)];
      if (!dft(B, false, v)) return -1;
      for (int k2 = 0; k2 < B; ++k2) y[place(k1, k2)] = v[k2];
    }
  } else {
    for (int k1 = 0; k1 < A; ++k1) {
      for (int k2 = 0; k2 < B; ++k2) v[k2] = x[place(k1, k2)];
      if (!dft(B, true, v)) return -1;
      for (int j = 0; j < B; ++j) mid[between(k1, j)] = v[j];
    }
    for (int j = 0; j < B; ++j) {
      for (int k1 = 0; k1 < A; ++k1) v[k1] = k1 ? cmul(mid[between(k1, j)], conj(w[k1 * B + j])) : mid[between(0, j)];
      if (!dft(A, true, v)) return -1;
      for (int r = 0; r < A; ++r) y[j + B * r] = v[r];
    }
  }
  return 0;
}

}  // extern "C"
