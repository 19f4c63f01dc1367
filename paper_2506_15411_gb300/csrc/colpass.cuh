// colpass.cuh -- the y and z passes of axes that split into two radices, n = A B, on column tiles.
//
//   y pass:  W_c <- FFT_y(W_c) or IFFT_y(W_c), one (component, z) plane x TX columns per tile
//   z pass:  W <- IFFT_z( G(p) FFT_z(W) ), the three components of one y row x TX columns,
//            G(p) the dyadic Green's function of curl curl - kt2, scaled by 1/N (green.cuh)
// (the k-space steps of the vector CBS of refs. [25], [26] of arXiv 2506.15411.)
//
// i = j + B r (j < B, r < A).  Step 1 of the forward transform: a thread takes one column's A
// values over r, output k1 times w_n^{j k1}; step 2: a thread takes the B values over j of one k1,
// output k2 is frequency k1 + A k2.  The inverse runs them backwards.  Both work in place: the
// value (k1, j) or (k1, k2) sits in row k1 B + (j ^ s), s = k1 & 1 for tiles of 8 columns and
// even B, else 0.  A row of 8 columns is half of the 32 banks; the swap puts two neighbouring k1 of
// step 2 into different halves.  Step 1 then writes rows that its neighbour j ^ 1 reads, which is
// in the same warp: a warp barrier between its loads and its stores is enough.  In the z pass
// step 2 runs forward, applies G and runs back on the three components in registers.
//
// A block is persistent: NG groups of GT threads, each with a named barrier and its own tile, and
// a warp that moves the tiles through a ring of S sets with the Tensor Memory Accelerator; a group
// neither waits for its stores nor meets at a barrier between tiles.  Small y tiles (below 24 KB)
// are stored by the group's first warp instead, which need not take turns with the other groups'
// stores (128^3: 0.0225 -> 0.0184 ms; the other way 256 x 256 x 192: 0.104 -> 0.099).
//
// Bounds and figures (ms, one GB300; staged passes of yz_kernels.cuh -> these).  y, 48 bytes a
// voxel, is bound by memory on large grids: 640 x 640 x 336 1.155 -> 1.09 (6.06 TB/s, 0.89 of a
// copy), 384 x 384 x 256 0.290 -> 0.294, 175 x 175 x 198 0.070 -> 0.051, 104 x 104 x 120 (a factor
// 13) 0.039 -> 0.0167, 128^3 0.030 -> 0.0205.  z, also 48 bytes, by instruction issue and shared
// memory, about half of each busy: 640 x 640 x 336 1.88 -> 1.35 (0.72 of a copy), 384 x 384 x 256
// 0.616 -> 0.342 (0.78), 275 x 275 x 315 0.371 -> 0.293, 256 x 256 x 192 0.165 -> 0.112 (0.80),
// 128^3 0.045 -> 0.0264.  The staged passes took three to four stages each way, a barrier and a
// trip through shared memory each, with offsets computed at run time.
#pragma once
#include <algorithm>
#include <utility>

#include "axis_plan.h"
#include "cbs_internal.h"
#include "fft_ip.cuh"
#include "green.cuh"
#include "tma.cuh"

namespace cbs {

namespace colk {

enum Kind { kYFwd = 0, kYInv = 1, kZ = 2 };

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void named_sync(int id, int count) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// Step 1 on NCOMP components of a tile: INV = false the forward's first step, else the inverse's
// last.  cs: component stride.
template <int A, int B, int TX, int NCOMP, int GT, bool INV>
__device__ __forceinline__ void col_step1(float2* buf, int cs, const float2* tw, int lt) {
  constexpr int items = NCOMP * TX * B;
  constexpr bool SW = TX == 8 && B % 2 == 0;
#pragma unroll 1
  for (int k0 = 0; k0 < items; k0 += GT) {
    if (items % GT && k0 + (lt & ~31) >= items) break;   // (a whole warp)
    const bool on = items % GT == 0 || k0 + lt < items;
    const int k = on ? k0 + lt : items - 1;   // an idle thread reads the last item and stores nothing
    const int col = k % TX, rest = k / TX;
    const int c = NCOMP > 1 ? rest / B : 0, j = NCOMP > 1 ? rest - c * B : rest;
    float2* const even = buf + c * cs + j * TX + col;
    float2* const odd = SW ? buf + c * cs + (j ^ 1) * TX + col : even;   // rows of odd k1
    const float2* const w = tw + j;
    float2 v[A];
#pragma unroll
    for (int r = 0; r < A; ++r) v[r] = (INV && SW && (r & 1) ? odd : even)[r * B * TX];
    if constexpr (INV) {
#pragma unroll
      for (int r = 1; r < A; ++r) {
        v[r] = cmul(v[r], ip_conj(w[r * B]));
        if (r % 8 == 0) asm volatile("" ::: "memory");   // (keeps the twiddles of a few products in registers, not all)
      }
    }
    DFT<A, INV>::run(v);
    if constexpr (SW) __syncwarp();
    if constexpr (!INV) {
#pragma unroll
      for (int r = 1; r < A; ++r) {
        v[r] = cmul(v[r], w[r * B]);
        if (r % 8 == 0) asm volatile("" ::: "memory");
      }
    }
    if (on) {
#pragma unroll
      for (int r = 0; r < A; ++r) (!INV && SW && (r & 1) ? odd : even)[r * B * TX] = v[r];
    }
  }
}

// Step 2 of a y tile.
template <int A, int B, int TX, int GT, bool INV>
__device__ __forceinline__ void col_step2(float2* buf, int lt) {
  constexpr int items = TX * A;
  constexpr bool SW = TX == 8 && B % 2 == 0;
#pragma unroll 1
  for (int k = lt; k < items; k += GT) {
    const int col = k % TX, k1 = k / TX;
    float2* const q = buf + k1 * B * TX + col;
    const int sw = SW ? (k1 & 1) * TX : 0;
    float2* const qe = q + sw;   // even j: row j ^ s
    float2* const qo = q - sw;   // odd j
    float2 v[B];
#pragma unroll
    for (int j = 0; j < B; ++j) v[j] = (j & 1 ? qo : qe)[j * TX];
    DFT<B, INV>::run(v);
#pragma unroll
    for (int j = 0; j < B; ++j) (j & 1 ? qo : qe)[j * TX] = v[j];
  }
}

template <int N, int KIND>
__global__ void __launch_bounds__(col_plan(N, KIND == kZ ? 3 : 1).threads(), 1)
    k_col(const __grid_constant__ CUtensorMap tm, const IterArgs a) {
  constexpr ColPlan CP = col_plan(N, KIND == kZ ? 3 : 1);
  constexpr int A = CP.A, B = N / CP.A, TX = CP.tx, GT = CP.gt, NG = CP.groups, NCOMP = KIND == kZ ? 3 : 1;
  constexpr bool COPY = KIND == kZ || N * TX * (int)sizeof(float2) >= 24000;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const ColShape& sh = KIND == kZ ? a.zc : a.yc;
  const int S = sh.sets, box = sh.box, nbox = sh.nbox;
  const int cs = nbox * box * TX;             // component stride
  const int tileN = NCOMP * cs;
  float2* const buf0 = reinterpret_cast<float2*>(smem_raw);   // S x [NCOMP][rows][TX]
  float2* const tw = buf0 + S * tileN;
  const int twb = KIND == kZ ? a.twbz : a.twby;
  float2* const pqz = tw + twb / sizeof(float2);              // z pass: wave numbers of k1 + A k2
  uint64_t* const full = reinterpret_cast<uint64_t*>(pqz + (KIND == kZ ? a.pqbz / (int)sizeof(float2) : 0));
  uint64_t* const done = full + S;
  uint64_t* const tbar = done + S;
  volatile int* const flags = reinterpret_cast<volatile int*>(tbar + 1);   // a wait gave up
  volatile int* const issued = flags + 1;                                    // tiles issued so far
  int* const bad = reinterpret_cast<int*>(tbar + 1) + 2;                     // tiles misaligned
  const int nxt = (a.nx + TX - 1) / TX;
  const int ntiles = KIND == kZ ? nxt * a.ny : nxt * a.nz * 3;
  const int G = KIND == kZ ? a.grid_z : a.grid_y;
  const MemberBlock mb = member_block(blockIdx.x, G);
  const int c0 = 3 * a.mem[mb.j].seat;   // the request's first component in the tensor map
  if (mb.b >= ntiles) return;
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid == 0) {
    *bad = (smem_u32(buf0) & 127u) ? 1 : 0;
    if (*bad) atomicExch(a.err, kErrMisaligned);
    *flags = 0;
    *issued = 0;
    for (int i = 0; i < S; ++i) {
      mbar_init(full + i, 1);
      mbar_init(done + i, COPY ? GT / 32 : 1);
    }
    mbar_init(tbar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (*bad) return;
  launch_dependents();

  const int n = (ntiles - mb.b + G - 1) / G;   // tiles of the block: mb.b, mb.b + G, ...

  // coordinates of tile t: x of its first column, its (z, component) or its row y
  auto y_tile = [&](int t, int& xt, int& z, int& c) {
    xt = t % nxt;
    const int r = t / nxt;
    z = r % a.nz;
    c = r / a.nz;
  };

  // A wait that gives up records the error and raises the block's flag.  The groups' later waits of
  // the block then return at once and every thread runs on through the same barriers (on stale
  // data; the host drops the result).  The copying warp stops: a set that was passed on unwaited for
  // may still have its copy under way, and its mbarrier cannot be armed for another.  Then it waits
  // until all it has loaded has landed, as the block may not end before; else every tile has been
  // waited for by the time the last one is done.  Where it does not see the last ones (small y tiles),
  // the groups do so too: either the flag was up by its last load, or that load counted before.
  auto give_up = [&] {
    *flags = 1;
    atomicExch(a.err, kErrTmaTimeout);
  };
  auto landed = [&] {
    const int sent = *issued;
    settle(full, S, max(0, sent - S), sent - 1);
    mbar_wait(tbar, 0);
  };
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    if (!*flags && !mbar_wait(bar, parity, a.wait_limit)) give_up();
  };

  if (tid >= NG * GT) {
    // the copying warp: loads the first S tiles; then, tile by tile, stores one that is done and,
    // once tile i (or, with sets to spare, the one before it) has been read out of its set, loads
    // the next tile into that set
    if (lane == 0) {
      mbar_arrive_expect_tx(tbar, twb + (KIND == kZ ? a.pqbz : 0));
      const int phase = twiddle_phase(a, a.mem[mb.j]);
      bulk_load(tw, KIND == kZ ? a.twz + phase * a.twsz : a.twy + phase * a.twsy, twb, tbar);
      if (KIND == kZ) bulk_load(pqz, a.pqz, a.pqbz, tbar);
    }
    const uint32_t bytes = (uint32_t)(tileN * sizeof(float2));
    auto load = [&](int t, int k) {
      if (lane == 0) {
        mbar_arrive_expect_tx(full + k, bytes);
        __threadfence_block();
        *issued = *issued + 1;
      }
      __syncwarp();
      float2* const dst = buf0 + k * tileN;
      if constexpr (KIND == kZ) {
        const int xt = t % nxt, y = t / nxt, yb = y / a.yblk, yi = y - yb * a.yblk;
        for (int i = lane; i < 3 * nbox; i += 32) {
          const int c = i / nbox, b = i - c * nbox;
          tma_load_5d(dst + c * cs + b * box * TX, &tm, xt * TX, yi, b * box, yb, c0 + c, full + k);
        }
      } else {
        int xt, z, c;
        y_tile(t, xt, z, c);
        for (int b = lane; b < nbox; b += 32)
          tma_load_5d(dst + b * box * TX, &tm, xt * TX, 0, z, b, c0 + c, full + k);
      }
    };
    // (whoever passed a set on without its wait has raised the flag before, and then this gives up)
    auto tile_done = [&](int k, uint32_t ph) { return warp_wait<true>(done + k, ph, flags, a.err, a.wait_limit); };
    bool ok = true;
    wait_for_previous();
    for (int i = 0; i < min(S, n); ++i) load(mb.b + i * G, i);
    if constexpr (!COPY) {
      int k = 0;
      uint32_t ph = 0;
      for (int i = S; i < n; ++i) {
        ok = tile_done(k, ph);
        if (!ok) break;
        load(mb.b + i * G, k);
        if (++k == S) {
          k = 0;
          ph ^= 1u;
        }
      }
      if (!ok || *flags) landed();
      return;
    }
    const int lag = S >= NG + 2 ? 1 : 0;
    int k = 0, kl = 0;   // sets of tile i and of the next tile to load
    uint32_t ph = 0;
    for (int i = 0; i < n; ++i) {
      const int t = mb.b + i * G;
      ok = tile_done(k, ph);
      if (!ok) break;
      const float2* const src = buf0 + k * tileN;
      if constexpr (KIND == kZ) {
        const int xt = t % nxt, y = t / nxt, yb = y / a.yblk, yi = y - yb * a.yblk;
        for (int m = lane; m < 3 * nbox; m += 32) {
          const int c = m / nbox, b = m - c * nbox;
          tma_store_5d(&tm, xt * TX, yi, b * box, yb, c0 + c, src + c * cs + b * box * TX);
        }
      } else {
        int xt, z, c;
        y_tile(t, xt, z, c);
        for (int b = lane; b < nbox; b += 32) tma_store_5d(&tm, xt * TX, 0, z, b, c0 + c, src + b * box * TX);
      }
      bulk_commit();
      if (lag) bulk_wait_read_1();
      else bulk_wait_read_all();
      __syncwarp();
      const int next = i - lag + S;
      if (i >= lag && next < n) {
        load(mb.b + next * G, kl);
        if (++kl == S) kl = 0;
      }
      if (++k == S) {
        k = 0;
        ph ^= 1u;
      }
    }
    if (!ok) landed();
    bulk_wait_all();
    return;
  }

  const int g = tid / GT, lt = tid - g * GT;
  auto gsync = [&] { named_sync(1 + g, GT); };
  wait(tbar, 0);
  float2 kt2 = make_float2(0.f, 0.f);
  if constexpr (KIND == kZ) kt2 = a.mem[mb.j].kt2;
#pragma unroll 1
  for (int i = g; i < n; i += NG) {
    const int t = mb.b + i * G, u = i / S, k = i - u * S;
    // the set's use u is armed once the tile counts as issued: before that its mbarrier may still
    // be two phases back, where the parity alone would let the wait through
    for (unsigned left = a.wait_limit; *issued <= i && !*flags; __nanosleep(32))
      if (left-- <= 1) give_up();
    wait(full + k, (uint32_t)(u & 1));
    float2* const cur = buf0 + k * tileN;
    if constexpr (KIND == kYFwd) {
      col_step1<A, B, TX, 1, GT, false>(cur, cs, tw, lt);
      gsync();
      col_step2<A, B, TX, GT, false>(cur, lt);
    } else if constexpr (KIND == kYInv) {
      col_step2<A, B, TX, GT, true>(cur, lt);
      gsync();
      col_step1<A, B, TX, 1, GT, true>(cur, cs, tw, lt);
    } else {
      // step 2's items of a thread are all in column lt mod TX (GT is a multiple of TX)
      const float2 px = __ldg(&a.pqx[(t % nxt) * TX + lt % TX]);
      const float2 py = __ldg(&a.pqy[t / nxt]);
      col_step1<A, B, TX, 3, GT, false>(cur, cs, tw, lt);
      gsync();
      constexpr bool SW = TX == 8 && B % 2 == 0;
      const GreenColumn col = green_column(px, py, kt2);
#pragma unroll 1
      for (int m = lt; m < TX * A; m += GT) {
        const int k1 = m / TX;
        float2* const q = cur + k1 * B * TX + m % TX;
        const int sw = SW ? (k1 & 1) * TX : 0;
        float2* const qe = q + sw;
        float2* const qo = q - sw;
        float2 v[3][B];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
#pragma unroll
          for (int j = 0; j < B; ++j) v[c][j] = (j & 1 ? qo : qe)[c * cs + j * TX];
          DFT<B, false>::run(v[c]);
        }
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2)
          green(col, pqz[k1 + A * k2], kt2, a.invN, a.invN_rest, v[0][k2], v[1][k2], v[2][k2]);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          DFT<B, true>::run(v[c]);
#pragma unroll
          for (int j = 0; j < B; ++j) (j & 1 ? qo : qe)[c * cs + j * TX] = v[c][j];
        }
      }
      gsync();
      col_step1<A, B, TX, 3, GT, true>(cur, cs, tw, lt);
    }
    fence_async_smem();
    if constexpr (COPY) {
      __syncwarp();
      if (lane == 0) mbar_arrive(done + k);
    } else {
      // the group's first warp waits for the others, which go on to their next tile, and stores
      if (lt >= 32) {
        asm volatile("bar.arrive %0, %1;" ::"r"(8 + g), "r"(GT) : "memory");
      } else {
        named_sync(8 + g, GT);
        int xt, z, c;
        y_tile(t, xt, z, c);
        for (int b = lane; b < nbox; b += 32) tma_store_5d(&tm, xt * TX, 0, z, b, c0 + c, cur + b * box * TX);
        bulk_commit();
        bulk_wait_read_all();
        __syncwarp();
        if (lane == 0) mbar_arrive(done + k);
      }
    }
  }
  if constexpr (!COPY) {
    if (*flags) landed();
    bulk_wait_all();
  }
}

}  // namespace colk

using ColKernel = void (*)(const CUtensorMap, const IterArgs);

// The kernels of an axis length (null: no such split), in parts n = part mod kColParts, each in a
// translation unit of its own (col_p*.cu).
constexpr int kColParts = 16;
struct ColKernels {
  ColKernel yfwd, yinv, z;
};

template <int N>
inline bool col_entry(int n, ColKernels& k) {
  if constexpr (N >= 4 && N <= 1024) {
    if (n == N) {
      if constexpr (col_plan(N, 1).A > 0) {
        k.yfwd = colk::k_col<N, colk::kYFwd>;
        k.yinv = colk::k_col<N, colk::kYInv>;
      }
      if constexpr (col_plan(N, 3).A > 0) k.z = colk::k_col<N, colk::kZ>;
    }
  }
  return n == N;
}
template <int PART, int... I>
inline ColKernels col_part(int n, std::integer_sequence<int, I...>) {
  ColKernels k{nullptr, nullptr, nullptr};
  (col_entry<PART + kColParts * I>(n, k) || ...);
  return k;
}
#define CBS_COL_PART(PART)                                                             \
  ColKernels col_kernels_##PART(int n) {                                               \
    return col_part<PART>(n, std::make_integer_sequence<int, 1024 / kColParts + 1>{}); \
  }

}  // namespace cbs
