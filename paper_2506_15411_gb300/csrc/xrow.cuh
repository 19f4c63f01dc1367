// xrow.cuh -- the x passes of axes that split into two radices, nx = A B: one warp owns whole rows.
//
//   first:    W_c = FFT_x(V E_c + S_c)                                  (a series' first x pass)
//   update:   W_c = IFFT_x(W_c);  delta_c = gamma (E_c - W_c);  E_c -= delta_c;  sum |delta|^2
//             (FP64);  then W_c = FFT_x(V E_c + S_c) of the next iteration, on the same tile
// (the update of the preconditioned series, refs. [25], [26] of arXiv 2506.15411).
//
// x = j + B r (j < B, r < A).  Forward: lane j transforms its A values over r, multiplies output
// k1 by w_n^{j k1}; lane k1 then transforms the B values over j, and output k2 is frequency
// k1 + A k2, stored there: the x spectrum in W is in natural order.  The inverse runs the same two
// steps backwards, and its second step, the update and the forward's first step work on one
// lane's A values in registers.  Both radices are at most 32, so a row's values of one step are
// in one warp's registers at once: a step reads all of them before it writes any, and the rows
// need neither a block barrier nor a scratch tile.  Between the two steps a row is kept as
// [k1][j] with row pitch P = 2 mod 4 (in complex values), so that lanes over j (8-byte accesses)
// and lanes over k1 (16-byte accesses at stride P) are both free of bank conflicts; the memory
// side of either step has lanes over consecutive elements.
//
// A block is persistent: T teams of three warps, one warp per field component, and a producer
// warp that keeps S tiles of rpb rows (W, E of three components, V) in flight or in hand.  A
// team's warps meet only at the mbarriers of their tile; each warp stores its own component.  A
// wait that gives up does so for its whole warp and raises the block's flag, at which the others give
// up too; all meet at the block's end, the producer once its copies have landed.
//
// Bound by memory: 104 bytes a voxel.  The staged pass (xpass.cu) spent its time at barriers and
// on shared memory, which its three or four stages cross 17 times per value, and on their bank
// conflicts; this one crosses it 13 times with two fifths of the conflicts (275 x 275 x 315: 47 ->
// 19 million; a quarter on rows of 640).  Update pass, staged -> rows (ms, one GB300):
// 640 x 640 x 336 2.91 -> 2.13 (6.7 TB/s, 0.99 of a copy), 384 x 384 x 256 0.966 -> 0.614 (0.94),
// 275 x 275 x 315 0.649 -> 0.383 (0.95), 256 x 256 x 192 0.356 -> 0.220 (0.88), 175 x 175 x 198
// 0.163 -> 0.109 (0.85), 192 x 192 x 128 0.128 -> 0.084 (0.86), 128^3 0.076 -> 0.047; 64^3 0.0214
// -> 0.0184 (latency of one to three tiles a block).
#pragma once
#include <algorithm>

#include "axis_plan.h"
#include "cbs_internal.h"
#include "fft_ip.cuh"
#include "tma.cuh"
#include "xpass_common.cuh"

namespace cbs {

namespace xrow {

constexpr int kRowThreads = 512;   // most threads of a block: five teams and the producer warp

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Step 2 of nr rows at `w` (row pitch ld): inverse (INV) reads frequency k1 + A k2 and writes
// [k1][j]; forward reads [k1][j] and writes the frequencies.  R = B.
template <int A, int B, bool INV>
__device__ __forceinline__ void row_step2(float2* w, int ld, int nr, int lane) {
  constexpr int R = B, P = row_pitch(B);
  constexpr int per = 32 / A;              // rows of a round
  const int lr = lane / A, k1 = lane - lr * A;
#pragma unroll 1
  for (int r0 = 0; r0 < nr; r0 += per) {
    const bool on = lr < per && r0 + lr < nr;
    float2* row = w + (on ? r0 + lr : 0) * ld;   // (an idle lane reads the first row and stores nothing)
    float2* f = row + k1;
    float2* x = row + k1 * P;
    float2 v[R];
    if constexpr (INV) {
#pragma unroll
      for (int k = 0; k < R; ++k) v[k] = f[k * A];
    } else {
      const float4* x4 = reinterpret_cast<const float4*>(x);
#pragma unroll
      for (int j = 0; j < R / 2; ++j) {
        const float4 u = x4[j];
        v[2 * j] = make_float2(u.x, u.y);
        v[2 * j + 1] = make_float2(u.z, u.w);
      }
      if constexpr (R % 2) v[R - 1] = x[R - 1];
    }
    DFT<R, INV>::run(v);
    __syncwarp();
    if (on) {
      if constexpr (INV) {
        float4* x4 = reinterpret_cast<float4*>(x);
#pragma unroll
        for (int j = 0; j < R / 2; ++j) x4[j] = make_float4(v[2 * j].x, v[2 * j].y, v[2 * j + 1].x, v[2 * j + 1].y);
        if constexpr (R % 2) x[R - 1] = v[R - 1];
      } else {
#pragma unroll
        for (int k = 0; k < R; ++k) f[k * A] = v[k];
      }
    }
    __syncwarp();
  }
}

// The x pass.  mode 0: the update pass.  1: form V E + S and transform it (the same code with W
// and 1 / epsilon taken as 0, which leaves E as it is).  2: the same for E = 0, reading nothing.
template <int A, int B>
__global__ void __launch_bounds__(kRowThreads, 1) k_xrow(const IterArgs a, const int mode) {
  constexpr int P = row_pitch(B);
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int rpb = a.xr.rpb, S = a.xr.sets, T = a.xr.teams;
  const int ldw = a.xr.ldw, lde = a.xr.lde;   // row pitches of W, and of E and V, in a tile
  const int rows = a.ny * a.nz, ntiles = (rows + rpb - 1) / rpb;
  const int G = a.grid_x;
  const int set = rpb * (3 * ldw + 4 * lde);
  float2* const set0 = reinterpret_cast<float2*>(smem_raw);
  float2* const tw = set0 + S * set;
  uint64_t* const full = reinterpret_cast<uint64_t*>(tw + a.twbx / sizeof(float2));   // [S]
  uint64_t* const empty = full + S;                                                   // [S]
  uint64_t* const tbar = empty + S;
  volatile int* const failed = reinterpret_cast<volatile int*>(tbar + 1);   // a wait gave up
  volatile int* const issued = failed + 1;                                  // tiles of the block issued so far
  int* const bad = reinterpret_cast<int*>(tbar + 1) + 2;                    // tiles misaligned

  const MemberBlock mb = member_block(blockIdx.x, G);
  const Member& mem = a.mem[mb.j];
  const size_t so = (size_t)mem.seat * 3 * a.Nw;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float acc = 0.f;
  if (mb.b < ntiles) {
    if (tid == 0) {
      *bad = (smem_u32(set0) & 127u) ? 1 : 0;
      if (*bad) atomicExch(a.err, kErrMisaligned);
      *failed = 0;
      for (int i = 0; i < S; ++i) {
        mbar_init(full + i, 1);
        mbar_init(empty + i, 3);
      }
      mbar_init(tbar, 1);
      *issued = 0;
      fence_mbar_init();
    }
    __syncthreads();
    if (*bad) return;
    launch_dependents();
    const uint32_t rb = (uint32_t)(((a.nx + 1) & ~1) * sizeof(float2));   // bytes of a row copy
    if (warp == 3 * T) {
      // producer: tile i of the block into set i mod S once the tile before it there is done
      const float2* const E = a.E + so;
      const float2* const W = a.W + so;
      const float2* const V = a.V + (size_t)mem.seat * a.Nw;
      if (lane == 0) {
        mbar_arrive_expect_tx(tbar, a.twbx);
        bulk_load(tw, a.twx + twiddle_phase(a, mem) * a.twsx, a.twbx, tbar);
      }
      wait_for_previous();
      int k = 0, n = 0;
      uint32_t ph = 1;   // a fresh mbarrier passes a wait for the phase before its first
      for (int tile = mb.b; tile < ntiles; tile += G) {
        if (!warp_wait(empty + k, ph, failed, a.err, a.wait_limit)) break;
        const int r0 = tile * rpb, nr = min(rpb, rows - r0);
        if (lane == 0) {
          mbar_arrive_expect_tx(full + k, (mode == 0 ? 7 : (mode == 1 ? 4 : 0)) * nr * rb);
          __threadfence_block();
          *issued = ++n;
        }
        __syncwarp();
        float2* const w = set0 + k * set;
        float2* const e = w + 3 * rpb * ldw;
        for (int i = lane; mode < 2 && i < 7 * nr; i += 32) {
          const int arr = ip_div(i, 1.0f / (float)nr), r = i - arr * nr;   // W 0..2, E 3..5, V 6
          const size_t g = (size_t)(r0 + r) * a.nxp;
          if (arr < 3) {
            if (mode == 0) bulk_load(w + (arr * rpb + r) * ldw, W + arr * a.Nw + g, rb, full + k);
          } else if (arr < 6) {
            bulk_load(e + ((arr - 3) * rpb + r) * lde, E + (arr - 3) * a.Nw + g, rb, full + k);
          } else {
            bulk_load(e + (3 * rpb + r) * lde, V + g, rb, full + k);
          }
        }
        if (++k == S) {
          k = 0;
          ph ^= 1u;
        }
      }
      // no copy may be under way when the sums below go over the tiles, or the block ends: a team
      // that gave up has not waited for its own
      settle(full, S, max(0, n - S), n - 1);
      mbar_wait(tbar, 0);
      __syncwarp();
    } else {
      const int team = warp / 3, c = warp - 3 * team;
      const int skind = mem.src.kind, splane = skind == 1 ? mem.src.pz : mem.src.zp;
      float2 amp = make_float2(0.f, 0.f);
      if (skind != 2) amp = (skind == 1 && mem.src.amp_dev) ? mem.src.amp_dev[c] : mem.src.amp[c];
      const float ie = mode ? 0.f : mem.inv_eps;
      const RowDecode rowdec = row_decode(a);
      float2* const Eg = a.E + so + c * a.Nw;
      float2* const Wg = a.W + so + c * a.Nw;
      constexpr int per = 32 / B;   // rows of a round of step 1
      const int lr = lane / B, j = lane - lr * B;
      bool ok = warp_wait(tbar, 0, failed, a.err, a.wait_limit);
#pragma unroll 1
      for (int i = team, tile = mb.b + team * G; ok && tile < ntiles; i += T, tile += T * G) {
        const int u = i / S, k = i - u * S;
        // the set's use u is armed once the tile counts as issued: before that its mbarrier may
        // still be two phases back, where the parity alone would let the wait through
        bool on = *issued > i;
        for (unsigned left = a.wait_limit; !on && !*failed && left > 0; --left) {
          __nanosleep(32);
          on = *issued > i;
        }
        if (!__all_sync(0xffffffffu, on)) {
          if (lane == 0) {
            *failed = 1;
            atomicExch(a.err, kErrTmaTimeout);
          }
          break;
        }
        if (!warp_wait(full + k, (uint32_t)(u & 1), failed, a.err, a.wait_limit)) break;
        const int r0 = tile * rpb, nr = min(rpb, rows - r0);
        float2* const w = set0 + k * set + c * rpb * ldw;
        float2* const e = set0 + k * set + 3 * rpb * ldw + c * rpb * lde;
        const float2* const v = set0 + k * set + 3 * rpb * (ldw + lde);
        if (mode == 0) row_step2<A, B, true>(w, ldw, nr, lane);
        constexpr int R = A;
#pragma unroll 1
        for (int q0 = 0; q0 < nr; q0 += per) {
          if (!(lr < per && q0 + lr < nr)) continue;
          const int row = q0 + lr;
          float2* const q = w + row * ldw + j;
          float2* const er = e + row * lde + j;
          const float2* const vr = v + row * lde + j;
          float2 x[R];
          if (mode == 0) {
            x[0] = q[0];
#pragma unroll
            for (int k1 = 1; k1 < R; ++k1) x[k1] = cmul(q[k1 * P], ip_conj(tw[k1 * B + j]));
            DFT<R, true>::run(x);
          } else {
#pragma unroll
            for (int r = 0; r < R; ++r) x[r] = make_float2(0.f, 0.f);
          }
          // the update at x = j + B r: delta = gamma (E - W), gamma = (i / epsilon) V;
          // E -= delta; then the next iteration's V E
          // (in chunks: the loads of a chunk before its stores)
          constexpr int U = 4;
          if (mode != 2) {
#pragma unroll
            for (int r0u = 0; r0u < R; r0u += U) {
              float2 vv[U], ec[U];
#pragma unroll
              for (int i2 = 0; i2 < U; ++i2)
                if (r0u + i2 < R) {
                  vv[i2] = vr[(r0u + i2) * B];
                  ec[i2] = er[(r0u + i2) * B];
                }
#pragma unroll
              for (int i2 = 0; i2 < U; ++i2)
                if (r0u + i2 < R) {
                  const int r = r0u + i2;
                  const float2 gm = make_float2(-vv[i2].y * ie, vv[i2].x * ie);
                  const float2 d = cmul(gm, csub(ec[i2], x[r]));
                  const float2 en = csub(ec[i2], d);
                  er[r * B] = en;
                  acc = fmaf(d.x, d.x, fmaf(d.y, d.y, acc));
                  x[r] = cmul(vv[i2], en);
                }
            }
          }
          int y, z;
          rowdec(r0 + row, y, z);
          if (skind == 0) {
            if (z == splane) {
#pragma unroll
              for (int r = 0; r < R; ++r) x[r] = cadd(x[r], amp);
            }
          } else if (skind == 1) {
            if (z == splane && y == mem.src.py) {
              const int px = mem.src.px;
#pragma unroll
              for (int r = 0; r < R; ++r)
                if (j + B * r == px) x[r] = cadd(x[r], amp);
            }
          } else {
            const float2* const us = mem.src.user + c * a.N + ((size_t)z * a.ny + y) * a.nx + j;
            const float sc = mem.src.user_scale;
#pragma unroll
            for (int r = 0; r < R; ++r) x[r] = cadd(x[r], cscale(__ldg(us + r * B), sc));
          }
          DFT<R, false>::run(x);
          q[0] = x[0];
#pragma unroll
          for (int k1 = 1; k1 < R; ++k1) q[k1 * P] = cmul(x[k1], tw[k1 * B + j]);
        }
        if (mode == 0) {
          fence_async_smem();
          __syncwarp();
          if (lane == 0) {
            for (int r = 0; r < nr; ++r) bulk_store(Eg + (size_t)(r0 + r) * a.nxp, e + r * lde, rb);
            bulk_commit();
          }
        }
        __syncwarp();
        row_step2<A, B, false>(w, ldw, nr, lane);
        fence_async_smem();
        __syncwarp();
        if (lane == 0) {
          for (int r = 0; r < nr; ++r) bulk_store(Wg + (size_t)(r0 + r) * a.nxp, w + r * ldw, rb);
          bulk_commit();
          bulk_wait_read_all();   // the set may be refilled once its rows have been read out
          mbar_arrive(empty + k);
        }
        __syncwarp();
      }
    }
  }
  if (mode == 0) {
    // the block's residual: the threads' sums through shared memory (every copy into it has landed
    // and every tile been read out of it by now), one warp adds them in FP64 in a fixed order
    float* const sums = reinterpret_cast<float*>(smem_raw);
    __syncthreads();
    sums[tid] = acc;
    __syncthreads();
    if (warp == 0) {
      double d = 0.0;
      for (int i = lane; i < blockDim.x; i += 32) d += (double)sums[i];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) d += __shfl_down_sync(0xffffffffu, d, off);
      if (lane == 0) *residual_slot(a, mem.seat, mb.b) = d;
    }
  }
  if (lane == 0) bulk_wait_all();
}

}  // namespace xrow

using RowKernel = void (*)(const IterArgs, const int);

// The kernel of an axis length (null: no split into two radices).  Lengths n = part mod kRowParts,
// each part in a translation unit of its own (xrow_p*.cu).
constexpr int kRowParts = 16;

template <int N>
inline bool row_entry(int n, RowKernel& k) {
  if constexpr (N <= 1024 && row_split(N) > 0)
    if (n == N) k = xrow::k_xrow<row_split(N), N / row_split(N)>;
  return n == N;
}
template <int PART, int... I>
inline RowKernel row_part(int n, std::integer_sequence<int, I...>) {
  RowKernel k = nullptr;
  (row_entry<PART + kRowParts * I>(n, k) || ...);
  return k;
}
#define CBS_ROW_PART(PART)                                                             \
  RowKernel row_kernel_##PART(int n) {                                                 \
    return row_part<PART>(n, std::make_integer_sequence<int, 1024 / kRowParts + 1>{}); \
  }

}  // namespace cbs
