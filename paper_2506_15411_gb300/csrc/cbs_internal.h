// cbs_internal.h -- structures shared by the host library and the CUDA kernels.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <cstddef>

#include "fft_ip.cuh"

namespace cbs {

constexpr int kBoxRows = 64;   // at most this many rows (y or z) per tensor-copy box

// Source term in the scaled units of the kernels (all k^2 quantities times pitch^2).
struct SourceArgs {
  int kind;               // 0 plane wave, 1 point, 2 user array
  float2 amp[3];          // plane wave: pol * (-2 i k_b pitch); point: pol * pitch^2
  int zp;                 // plane-wave sheet
  int px, py, pz;         // point-source voxel
  const float2* amp_dev;  // point source with amplitudes on the device (adjoint), or null
  const float2* user;     // user S [3][N]
  float user_scale;       // pitch^2
};

// Requests that share one launch: a plan's arrays (E, W, V) hold `seats` requests of the same
// grid side by side, and a launch iterates up to kMaxMembers of them, each with its own source
// and splitting (an array of Member in device memory, written before the launch).  A launch's
// grid is nmem times the per-request persistent grid; block b works for member b / grid, as
// block b mod grid of that request's own persistent grid, so every request's tiles, and the
// order of its residual sums, are the same in any launch.
constexpr int kMaxMembers = 8;
constexpr int kResidualSlots = 64;   // iterations whose residual partials are kept

struct Member {
  SourceArgs src;
  float inv_eps;          // 1 / epsilon (scaled)
  float2 kt2;             // k0^2 + i epsilon (scaled)
  int phase;              // of the twiddle tables at slot 0: iterations of its series before the block
  int seat;               // slice of the plan's arrays: E, W at + seat * 3 Nw; V at + seat * Nw
};

// Grids up to this many voxels launch an iteration's kernels overlapped: each may take up
// processors as the blocks of the one before leave them.  That saves 4 us an iteration where it
// lasts tens (64^3 32.2 -> 28.6 us, 128^3 96.0 -> 91.5, 192 x 192 x 128 193 -> 191), but the blocks
// then land on processors in any order, and neighbouring tiles, which share memory lines, on
// both dies: 175 x 175 x 198 284 -> 290 us, 640 x 640 x 336 5.7 -> 6.6 ms.  The members of a launch do
// not count: their tiles share no lines, and each brings a wave of blocks of its own (eight of
// 192 x 192 x 128, 32 iterations and half as many adjoints: 77.9 ms, plain launches 78.7; eight of 128^3
// 40.0, 40.7; eight of 112 x 108 x 96 26.8, 27.3; four of 160 x 150 x 140 30.1, 30.8; two 14.3, 14.3).
constexpr size_t kOverlapVoxels = 5000000;

// Launch a kernel that calls wait_for_previous() before it touches what the kernel before it in
// the stream wrote; overlap: it may start while that kernel's last blocks run.
template <class... P, class... Q>
cudaError_t launch_overlapped(void (*k)(P...), int grid, int threads, size_t smem, bool overlap, cudaStream_t s,
                              Q&&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = overlap ? 1 : 0;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = &at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, k, static_cast<Q&&>(args)...);
}

// Shapes of the x passes of an axis nx = A B (xrow.cu); A = 0: the staged passes (xpass.cu).
struct XRowShape {
  int A, B;               // radices: x = j + B r, frequency k1 + A k2
  int ldw, lde;           // row pitches of W, and of E and V, in a tile
  int rpb, sets, teams;   // rows of a tile, tiles in shared memory, teams of three warps
};

// Shapes of the column passes of an axis n = A B (colpass.cuh); sets = 0: the staged passes.
struct ColShape {
  int sets;               // tiles in shared memory
  int box, nbox;          // rows of a tensor-copy box, boxes of a component
  int threads, tx;
};

// Everything one CBS iteration needs (kernel parameters, by value).
struct IterArgs {
  int nx, ny, nz;
  size_t N;               // nx * ny * nz (fields E, V, sources: dense rows)
  int nxp;                // row pitch of the workspace W (multiple of 16 complex values)
  int yblk, nyb;          // y-blocked layout: blocks of yblk y rows (yblk divides ny), nyb blocks
  size_t Nw;              // nxp * ny * nz: component stride of W, E
  int yb, zb;             // rows per tensor-copy box along y and z
  int nyr, nzr;           // ny, nz rounded up to whole boxes (shared-memory rows of a tile)
  AxisIP ax, ay, az;      // in-place FFT plans (fft_ip.cuh)
  const float2* twx;      // per-stage twiddle tables; each 128-byte aligned, padded to n entries
  const float2* twy;
  const float2* twz;
  int twsx, twsy, twsz;   // from one phase's twiddles to the next (0: one table)
  int twbx, twby, twbz;   // bytes copied per table: n * 8 rounded up to a multiple of 16
  const float2* pqx;      // wave numbers (p, q) of each position of an axis' spectrum,
  const float2* pqy;      // padded with zeros to a multiple of 16 entries
  const float2* pqz;
  int pqbz;               // bytes of the z table the z pass copies (multiple of 16)
  float2* E;              // fields being iterated, [seats][3][nyb][nz][yblk][nxp] (plan-owned)
  float2* W;              // workspace, same layout
  const float2* V;        // potential [seats][nyb][nz][yblk][nxp], scaled
  int seats;              // requests the arrays hold
  int nmem;               // members of this launch (1 .. kMaxMembers)
  const Member* mem;      // their sources, splittings and seats (device memory)
  float invN, invN_rest;  // 1 / N, folded into the k-space multiply: invN (1 + invN_rest)
  double* partials;       // residual partial sums, [seat][kResidualSlots][grid_x]
  double* hist;           // hist[seat * hist_cap + slot] = sum |delta|^2 of this iteration
  int hist_cap;
  int slot;
  int* err;               // device error flag (a tensor-copy wait that timed out)
  unsigned wait_limit;    // polls after which a wait on a tile gives up
  // launch shapes
  XRowShape xr;
  ColShape yc, zc;
  int rpb;                // rows per tile, x passes
  int nset_x, nset_xf;    // buffer sets of the x passes (inverse + forward; first forward)
  int tx_y, tx_z;         // x-columns per tile, y and z passes
  int nbuf_y, nbuf_z;     // tile buffers of the pipelined y and z passes (2 to 4)
  int occ_y, occ_z;       // blocks per SM of the y and z kernels (2: radices <= 11, 64 registers)
  int maxr_x, maxr_z;     // largest radix of the x and z axes (selects the kernel build)
  int xgroups, zgroups;   // warp groups of the fused x and the z blocks (1 or 2)
  int grid_x, grid_xf, grid_y, grid_z;   // persistent grid sizes of one request (x inverse,
                                         // x forward, y, z); a launch has nmem times as many
};

// Block b of a launch: member b / G, block b mod G of that member's grid of G blocks.
struct MemberBlock {
  int j, b;
};
CBS_HD MemberBlock member_block(int block, int G) {
  const int j = block / G;
  return MemberBlock{j, block - j * G};
}

// The plan's arrays (W, the iterate E, V) store row (y, z) of a component at
//     ((y / yblk) * nz + z) * yblk + y mod yblk
// -- blocks of yblk consecutive y rows, z inside a block: a z column then visits rows yblk
// rows apart (instead of ny), and a y column runs in nyb stretches of yblk rows.  Long
// z strides of the plain [z][y] order slowed the z pass by half on a 640 x 640 plane.
CBS_HD size_t wrow(int y, int z, int nz, int yblk) {
  const int yb = y / yblk;
  return ((size_t)yb * nz + z) * yblk + (y - yb * yblk);
}

// The twiddle tables of this launch's iteration, for a member (axis_plan.h).
CBS_HD int twiddle_phase(const IterArgs& a, const Member& m) { return (a.slot + m.phase) % kTwiddlePhases; }

// Launchers (one per pass of an iteration); each returns the launch error.
cudaError_t launch_xpass_fwd(const IterArgs& a, bool zero, cudaStream_t s);   // W = FFTx(V E + S); zero: E is 0
cudaError_t launch_ypass(const CUtensorMap& tm, const IterArgs& a, bool inverse, cudaStream_t s);
cudaError_t launch_zpass_green(const CUtensorMap& tm, const IterArgs& a, cudaStream_t s);  // FFTz, G, IFFTz
cudaError_t launch_xpass_inv_fwd(const IterArgs& a, cudaStream_t s);  // IFFTx, update, residual, next FFTx

// Sum the residual partials of iterations slot0 .. slot0 + count - 1 (count <= kResidualSlots, none of
// them wrapped) of seats 0 .. seats - 1 into hist.
cudaError_t launch_residuals(const IterArgs& a, int slot0, int count, int seats, cudaStream_t s);

// Shared-memory bytes and threads of each pass for the plan's shapes.
size_t xpass_smem(const IterArgs& a);
int xpass_tiles(const IterArgs& a);
size_t xrow_smem(const IterArgs& a);
int xrow_tiles(const IterArgs& a);
cudaError_t launch_xrow(const IterArgs& a, int mode, cudaStream_t s);   // the x passes of nx = A B
cudaError_t xrow_set_smem_limit(int n, int bytes);
cudaError_t launch_col(const CUtensorMap& tm, const IterArgs& a, int kind, cudaStream_t s);   // y, inverse y, z
cudaError_t col_set_smem_limit(int n, bool z, int bytes);
cudaError_t yz_grid_sizes(IterArgs& a, int sms);   // sets grid_y, grid_z
cudaError_t x_grid_size(IterArgs& a, int sms);     // sets grid_x, grid_xf

// Set-up and gradient kernels (misc.cu).
// The splitting of a permittivity as the set-up kernels leave it on the device.
struct Splitting {
  double k0sq, eps;       // scaled k0^2 and epsilon
  int bad;                // a non-finite permittivity
  unsigned count;         // last-block counter (left at 0)
};
// xlo .. xhi - 1: the voxels along x outside the absorbing layers
cudaError_t launch_splitting(const float* eps, int nx, int ny, int nz, int xlo, int xhi, const double* sx, const double* sy,
                             const double* sz, int corner_max, double kv2, float* pmin, float* pmax, int* pbad,
                             double* part, int blocks, Splitting* sp, cudaStream_t s);
cudaError_t launch_build_v(const float* eps, int nx, int ny, int nz, int nxp, int yblk, int xlo, int xhi, const double* sx,
                           const double* sy, const double* sz, int corner_max, double kv2, const Splitting* sp,
                           float2* V, cudaStream_t s);
// A field between the caller's dense layout [3][nz][ny][nx] and the plan's y-blocked one
// (to_dense: plan -> dense); the row padding of the plan's copy is not written.
cudaError_t launch_field_layout(const float2* src, float2* dst, bool to_dense, int nx, int ny, int nz, int nxp,
                                int yblk, cudaStream_t s);
cudaError_t launch_adjoint_amp(const float2* E, size_t N, int nx, int ny, int x, int y, int z,
                               float scale, float2* amp, cudaStream_t s);
cudaError_t launch_gradient(const float2* E, const float2* Ea, size_t N, float coef, float* g,
                            cudaStream_t s);
cudaError_t launch_objective(const float2* E, size_t N, int nx, int ny, int x, int y, int z,
                             double* out, cudaStream_t s);

// Bounded-wait self-test (misc.cu): *err = 1 (tensor-copy wait timed out) after `limit` polls.
cudaError_t launch_wait_selftest(int* err, long long limit, cudaStream_t s);

// Inverse-design kernels on the thickness map (design.cu).
cudaError_t launch_mirror(const float* in, float* out, int nx, int ny, cudaStream_t s);
cudaError_t launch_filter(const float* in, float* out, int nx, int ny, const float* w, int R, int axis,
                          cudaStream_t s);
cudaError_t launch_height_to_eps(const float* heff, float* eps, int nx, int ny, int nz, int z_base, float inv_pitch,
                                 float eb, float de, int sms, cudaStream_t s);
cudaError_t launch_surface_grad(const float* g, const float* heff, float* out, int nx, int ny, int nz, int z_base,
                                float inv_pitch, float slope, cudaStream_t s);
cudaError_t launch_adam(float* h, const float* gh, float* m, float* v, int nx, int ny, double pitch_um,
                        double r2max, float alpha, float b1, float b2, float c1, float c2, float aeps, float hmax,
                        cudaStream_t s);

}  // namespace cbs
