// Handle of one lattice (shared by the library's CUDA translation units).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include "lbm_kernels.cuh"

namespace lbm {
// Cut of an nx x ny lattice into gx x gy tiles (tile b: columns [b nx / gx, (b + 1) nx / gx)),
// all at least four nodes wide and high unless the lattice itself is smaller.
struct ResPlan {
  int gx, gy;
  int wmax, hmax;    // largest tile
  int pitch;         // row pitch of a tile and its halo in shared memory
  int threads;       // of a block
  unsigned smem;     // dynamic shared memory of a block
  size_t words;      // 16-byte words of one parity of the exchange buffer, all tiles
  int steps;         // at most, of one launch
};
}  // namespace lbm

struct lb_handle {
  lb_params p;
  lb_derived d;
  void* f[2];
  int cur;
  void* scratch;
  size_t scratch_bytes;
  cudaStream_t stream;
  int64_t steps;
  int variant;  // LB_FUSED or LB_TWO_PASS
  int reduce_blocks;
  lbm::Strides st;        // population layout (planes or rows)
  bool use_tma;           // FP32 fused step with tensor-copy staging (interior tiles)
  int tma_grid;           // persistent grid of that kernel
  int tma_grid_auto;      // its default: resident capacity, at most the tile count
  unsigned* queue;        // tile tickets of the dynamic form (end of the scratch buffer), or null
  bool use_dyn;           // the tensor-copy step takes tiles by ticket (k_step_tma_dyn)
  int dyn_grid, dyn_grid_auto;
  CUtensorMap tmap[2];    // 3-D maps of f[0] and f[1]: (x, y, plane), rows layout (x, plane, y)
  int* wait_error;        // this handle's device word, set by a bounded wait that gave up
  int wait_slot;          // its index in the library's array of such words (-1: none taken)
  // Replay of runs of steps (lb_step): graphs of kStepGraph steps captured on an
  // internal stream, one per starting buffer, with the launch configuration they
  // were captured for; events order them after and before the caller's stream.
  cudaStream_t gstream;
  cudaEvent_t gev[2];
  cudaGraphExec_t graph[2];
  long long graph_cfg[2];
  bool graph_off;         // capture failed once: direct launches only
  // Resident run (lbm_resident.cu): many steps per launch on lattices that fit the SMs'
  // shared memory.
  bool use_res;
  bool plain_small;       // small enough for k_step_fused although tensor copies could serve it
  bool forced_dispatch;   // lb_set_tile_dispatch asked for a tensor-copy form
  bool forced_blocks;     // lb_set_step_blocks fixed its grid
  lbm::ResPlan res;
  int res_mode;           // lb_set_resident: -1 by rule, 0 never, 1 always
  int res_fit;            // resident runs of this lattice that fit the GPU side by side
  int64_t res_refuse;     // lb_resident_selftest: launches until one is taken for refused (-1: none)
  int res_dev;            // device
  bool res_live;          // the handle counts among those that step resident (res_enter)
  void* res_mail;         // exchange words (end of the scratch buffer)
  unsigned* step_word;    // device word with the step count a replayed FP16 graph seeds from
  bool overlap;           // the steps' launches may overlap their predecessor's end (lbm_launch.cuh)
  int graph_k;            // while capturing: the place of the launch in the graph (else -1)
  lbm::VCoef<float> cf;  // FP32 scalar (two-pass variant, moments)
  lbm::VCoef<lbm::f2> c2;     // FP32 pairs (fused variant)
  lbm::VCoef<double> cd;
  char err[512];
};

namespace lbm {
// 3-D tensor map of an FP32 (elem_bytes 4) or FP16 (2) population buffer, box =
// one plane window of the tensor-copy step: dimensions (x, y, plane) with row
// stride sx, or (x, plane, y) for the rows layout (sx = nx); false if the layout
// does not allow one (lbm_capi.cu).
bool encode_population_map(CUtensorMap* map, void* base, int nx, int ny, int sx, int elem_bytes = 4,
                           bool rows = false);
// 3-D map (x, y, plane) of `planes` FP32 planes of nx x ny, box cols x rows x 1
// (lbm_capi.cu); false if the buffer does not allow one.
bool encode_plane_map(CUtensorMap* map, const void* base, int nx, int ny, int planes, int cols, int rows);
// 4-D map (x, y, z, plane) of `planes` FP32 volumes of nx x ny x nz, box of cols x rows x
// 1 x 1 (lbm_capi.cu); false if the buffer does not allow one.
bool encode_volume_map(CUtensorMap* map, const void* base, int nx, int ny, int nz, int planes, int cols, int rows);
// Cut of a lattice for the resident run; false if it does not fit (lbm_resident.cu).
bool res_plan(int nx, int ny, int precision, ResPlan* out);
// Bytes of the exchange buffer (0 when no precision of this size runs resident).
size_t res_mail_bytes(int nx, int ny);
// Decides whether the handle can run resident with the exchange buffer `mail` (device
// memory of res_mail_bytes, 16-byte aligned, or null; its contents do not matter).
cudaError_t res_configure(lb_handle* h, void* mail);
// Counts the handle among those that step resident (its first call that is long enough),
// and takes it out again (lb_free).
void res_enter(lb_handle* h);
void res_leave(lb_handle* h);
// Streams of the handle's device that counted handles are bound to, its own included.
int res_streams(const lb_handle* h);
// Advances the handle's lattice by nsteps >= 2 steps and its counters with it; rec (or
// null): device memory that receives the states after every `every` steps.
// *done: the steps taken; fewer than nsteps if the device refused a launch, in which case the
// handle no longer runs resident.
cudaError_t res_run(lb_handle* h, int64_t nsteps, void* rec, int64_t every, int64_t* done);
// Device address of lb_reduce_static's static scratch on the current device
// (looked up once per device, which commits the array there; lbm_static.cu).
int static_scratch_address(lb_handle* h, void** out);
// Mean of the n doubles at x (device memory), summed in FP64 on `stream` with
// block partials written to `work` (device memory of work_bytes >= 8), folded on
// the host in a fixed order; synchronous.  cudaSuccess or the CUDA error
// (lbm_capi.cu).
cudaError_t device_mean(const double* x, size_t n, void* work, size_t work_bytes, cudaStream_t stream, double* mean);
}  // namespace lbm
