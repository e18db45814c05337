// lb_internal.h -- launchers shared between the translation units of the
// library (FP64 parity build, FP32 build, host API).  Not part of the ABI.
#pragma once

#include <cstddef>
#include <cstdint>
#include <vector>
#include <cuda.h>
#include <cuda_runtime.h>

namespace lbk {

// Arguments of the strip-sweep kernel (lb_sweep.cu).  The state buffers use
// the padded layout: plane q, interior site (x, y) at element
// q * plane + off + y * pitch + x, with 4 ghost columns and 4 ghost rows on
// each side.  FP32 storage: nine float planes at fout.  16-bit deviation
// storage: the rest population as one float plane at fout, the deviations
// d_i = f_i - r_i (i = 1..8) as eight 16-bit planes at fdev (same pitch,
// plane and offset, counted in 16-bit elements).
//
// Constants of the packed FP32 arithmetic, each twice (one per half of a
// pair): a pair instruction reads them as one 64-bit operand, and no
// instruction is spent on building the pair.
struct SweepConsts {
  // of the lattice
  float2 T, nb /* -b */, a, kappa, A0;
  float2 N, M, Q, R, m4QR /* -4 (Q + R) */;
  float2 th, g, om /* omega */, om1 /* 1 - omega */;
  float2 Aax /* A_ax / 9 */, Adg /* A_diag / 36 */;
  float2 r_sum;           // 16-bit storage: sum of the moving links' references
  float2 mwr_ax, mwr_dg;  // -omega r_ax, -omega r_dg
  // of the scheme
  float2 one, half, two, m6 /* -1/6 */, m24 /* -1/24 */, e8 /* 1/8 */, q4 /* 1/4 */, mq4;
  float2 third, mthird, twelfth, mtwelfth;
};
constexpr int kLatticeConsts = 19;  // the first of them, those of the lattice
struct SweepArgs {
  int nx, ny, walls;
  int pitch;
  long long plane, off;
  // tiles: nseg segments of seg_h rows by nstrips columns of tiles, base_w
  // wide (the first `extra` wider by the column quantum, the last narrower by
  // `pad`: nx rounded up to the quantum, minus nx)
  int seg_h, nseg, nstrips, base_w, extra, pad;
  SweepConsts k;
  float u_bot, u_top;
  float nmax;                  // 1/b (upper bound of a valid density)
  float ref_ax, ref_dg;        // reference populations r_i of the 16-bit format
  const float *sinx;
  const float *fin;            // the input state and its deviation planes
  const void *fdin;
  float *fout;
  void *fdev;
  double *partials;            // 4 doubles per CTA: mass, J_x, J_y, bad-site flag
  int records;                 // write the per-CTA records (0: skip them)
  unsigned wait_limit;         // looks at a copy's barrier before a wait of a single step gives up
  int *err;                    // set when a bounded wait gave up
  // Non-null (single-lattice launches with records only): the last CTA to
  // finish sums every CTA's record in a fixed order into total[0..4] --
  // mass, J_x, J_y, 1.0 if any record flags a bad site, 1.0 if *err is set
  // -- and resets *arrivals (a counter that is zero between launches).
  double *total;
  unsigned *arrivals;
  // Non-null: the same last CTA also writes {total[0..4], mon_step} here
  // (device address of a record in a mapped host ring).
  double *monitor;
  double mon_step;
};

// Looks at a barrier or a counter before a wait of the sweep kernels gives up.
constexpr unsigned kSweepWaitLimit = 1u << 22;

// Storage formats of the sweep kernel (values of lb_precision).
constexpr int kStoreF32 = 1, kStoreBF16 = 2, kStoreFP16 = 3;
// FP32 with a number of columns that is not a multiple of 4.
constexpr int kStoreF32Odd = 4;

// Whether the sweep kernel of storage `store` can run an nx x ny lattice
// (column quantum of its TMA boxes, ghost bands, 32-bit plane offsets).
bool sweep_supported(int store, int nx, int ny);
// (tau1 here and below: the form for relaxation time exactly 1, whose collision
// reads no populations; every lattice of the launch must have it)
cudaError_t sweep_prepare(int store, bool tau1, size_t *smem_bytes);
// Default tiling of the sweep kernel for an nx x ny lattice: the fewest strips
// and segments of 64 rows.
void sweep_plan(int store, int nx, int ny, int *nstrips, int *seg_h);
// Columns of tiles of a tiling with nstrips strips: one per strip, or, where a
// strip is wider than a tile can be, the fewest that cover the lattice.
int sweep_tile_cols(int store, int nx, int nstrips);
// Segment height that gives about as many tiles in all as `resident` warps
// want, for lattices of `cols` tile columns over ny rows (cols may sum over
// several lattices).
int sweep_seg_rule(double cols, int ny, int resident, bool batch = false);
// Sleep (ns) between two looks at a dependency in a launch of nitems tiles a
// step on a device that holds `resident` warps.
unsigned sweep_poll_ns(int nitems, int resident);
// Warps of the sweep kernel one SM holds (shared memory and registers).
int sweep_warps_per_sm(int store, bool tau1);
// Widths of nstrips strips (>= sweep_min_strips, the fewest a tiling may name) over nx columns: base_w or
// base_w + quantum, the first `extra` wider.
void sweep_strips(int store, int nx, int nstrips, int *base_w, int *extra);
int sweep_min_strips(int store, int nx);
// TMA descriptors of one padded state buffer with the boxes the kernel's
// ring expects (built next to the kernel so the two cannot differ).  FP32:
// one map of the nine planes (m1 is a copy).  16-bit storage: m0 maps the
// float rest plane at base, m1 the eight deviation planes that follow it.
cudaError_t sweep_make_maps(int store, void *base, int pitch, int ny, long long plane, CUtensorMap *m0,
                            CUtensorMap *m1);
// Bytes of one padded state buffer of the given storage.
size_t sweep_buffer_bytes(int store, long long plane);
cudaError_t launch_sweep(int store, bool tau1, const CUtensorMap &m0, const CUtensorMap &m1, const SweepArgs &A,
                         size_t smem, cudaStream_t st);

// Density and velocity u* of the state A.fin describes (maps m0, m1) into
// compact arrays n, ux, uy (each may be null; dtype 0 = double, 1 = float; host:
// they are page-locked host memory).
cudaError_t launch_sweep_moments(int store, const CUtensorMap &m0, const CUtensorMap &m1, const SweepArgs &A, void *n,
                                 void *ux, void *uy, int dtype, bool host, cudaStream_t st);

// Dependency lists of the tiles (CSR): tile a waits for the tiles
// idx[ofs[a] .. ofs[a+1]) before each step.  Tile = column + ncol * segment;
// `window` is the number of columns a tile is taken to read from its origin
// - 4 (kSweepWindow: what the kernel reads).
constexpr int kSweepWindow = 64;
void sweep_deps(int store, int nx, int ny, int walls, int ncol, int base_w, int extra, int seg_h, int window,
                std::vector<int> &ofs, std::vector<int> &idx);

// One CTA of the batched sweep: instance `inst`, its strip and segment, the
// index of its mass/momentum record in the instance's record array, and the
// parity of the instance's input buffer at kpar = 0.
struct BatchItem {
  int inst, strip, seg, rec, par0;
};
// Batched step over a work list.  args: 2 per instance (input buffer 0, 1);
// maps: 4 per instance ([input buffer][map], map 1 = deviation planes of
// 16-bit storage or a copy of map 0), 64-byte aligned device memory.
// (k: the consts of the scheme)
cudaError_t launch_sweep_batch(int store, bool tau1, const BatchItem *items, int nitems, const SweepArgs *args, const SweepConsts &k,
                               const CUtensorMap *maps, int kpar, int records, size_t smem, cudaStream_t st);
// Multi-step sweeps (one launch, many steps, per-item completion counters
// instead of a grid-wide barrier between steps).
// Item i of a step whose batch parity is kpar reads the input buffer
// items[i].par0 ^ kpar of its lattice; kpar = (kpar0 + k) & 1 at step k.
struct MultiArgs {
  int nitems;
  int nsteps;
  int kpar0;
  unsigned epoch;       // value of every done[] counter at launch
  unsigned *done;       // one per item
  const int *dep_ofs;   // item i depends on dep_idx[dep_ofs[i] .. dep_ofs[i+1])
  const int *dep_idx;
  unsigned *next;       // ticket counter, zero at launch
  unsigned poll_ns;     // sleep between two looks at a counter (sweep_poll_ns)
};
// Outputs of the single-lattice multi-step kernel: the step that reads
// buffer b writes fout[b] (and fdev[b], the deviation planes of 16-bit
// storage); the last step's CTA records are summed into total[0..4] by the
// CTA that finishes last (arrival counter *arrivals, zero between
// launches).
struct MultiOut {
  float *fout[2];
  void *fdev[2];
  double *total;
  unsigned *arrivals;
  // Monitoring (mon_ring non-null): every step k writes its records into
  // slot k of mon_recs (4 doubles per tile) and counts on mon_arr[k]; the
  // CTA that finishes step k last adds them and writes the step's record
  // {mass, J_x, J_y, unstable, wait error, step number} at
  // mon_ring + 6 * ((mon_step0 + k) % mon_cap).
  double *mon_recs;
  unsigned *mon_arr;
  double *mon_ring;
  int mon_cap;
  long long mon_step0;
};
// One lattice, P.nsteps steps in one launch (P.kpar0 = the
// input buffer of the first step; items are the tiles in index order).
cudaError_t launch_sweep_multi(int store, bool tau1, const CUtensorMap (&maps)[2][2], const SweepArgs &A, const MultiArgs &P,
                               const MultiOut &Q, size_t smem, cudaStream_t st);
// P.nsteps batch steps in one launch; the mass / momentum records of the last
// step go to each instance's record array.
cudaError_t launch_sweep_batch_multi(int store, bool tau1, const BatchItem *items, const SweepArgs *args, const SweepConsts &k,
                                     const CUtensorMap *maps, const MultiArgs &P, size_t smem, cudaStream_t st);
// Copy the periodic images into the ghost band of `nplanes` planes of
// `elem_bytes`-byte elements (4 or 2).
cudaError_t launch_ghost_fill(void *f, int elem_bytes, int nplanes, int nx, int ny, int pitch, long long plane,
                              long long off, int walls, cudaStream_t st);
template <typename real_t>
struct StepArgs;

// One fused time step fin -> fout.
cudaError_t launch_step(const double *fin, double *fout, const StepArgs<double> &A, cudaStream_t st);
cudaError_t launch_step(const float *fin, float *fout, const StepArgs<float> &A, cudaStream_t st);

// Moments (n, u*) of the stored state; dtype 0 = double, 1 = float outputs.
cudaError_t launch_moments(const double *fin, const StepArgs<double> &A, void *n, void *ux,
                           void *uy, int dtype, cudaStream_t st);
cudaError_t launch_moments(const float *fin, const StepArgs<float> &A, void *n, void *ux,
                           void *uy, int dtype, cudaStream_t st);

// Equilibrium initial state from noise (mode 0) or device fields (mode 1).
cudaError_t launch_init(double *f, int nx, int ny, int pitch, long long plane, long long off, int mode, uint64_t seed, double rho_mean,
                        double amp, const double *rho0, const double *ux0, const double *uy0,
                        double T, cudaStream_t st);
// The same for FP32 and 16-bit lattices (lb_init.cu): the state buffer buf of
// storage `store` in one pass, its ghost band included.
struct InitState {
  int nx, ny, pitch;
  long long plane, off;
  int images;  // periodic images to write: 0 none (compact planes), 1 along x (walls), 2 along x and y
  uint64_t seed;
  double rho_mean, amp, T;
  const double *n0, *ux, *uy;  // density and velocity fields; n0 null: noise
  float ref_ax, ref_dg;
};
cudaError_t launch_init_f32(int store, void *buf, const InitState &I, cudaStream_t st);

}  // namespace lbk
