// D3Q19 form of the self-tuning-EOS multiphase lattice Boltzmann time step
// (Huang, Wu & Adams, arXiv:1809.02390, extended to three dimensions) and the
// lb_d3_* C ABI of include/lbm3d.h.
//
// The step kernel and its device code are in lbm3d_step.cuh.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "lbm3d.h"
#include "lbm_internal.h"
#include "lbm_handle.cuh"

#include "lbm3d_step.cuh"

namespace {

// Initial state at rest from FP64 densities: deviations of M^-1 m_eq(rho, 0).
// Invalid densities record the first offending node in bad[0] (not positive and
// finite) or bad[1] (vdW: rho >= 1/b).
template <typename T>
__global__ void k_d3_init(const double* __restrict__ rho0, T* __restrict__ f, int N, C3<double> c,
                          unsigned long long* bad) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  const double rho = rho0[n];
  if (!(rho > 0.0) || !isfinite(rho)) {
    atomicMin(bad, (unsigned long long)n);
    return;
  }
  if (c.eos == LB_EOS_VDW && !(c.b * rho < 1.0)) {
    atomicMin(bad + 1, (unsigned long long)n);
    return;
  }
  const double delta = rho - c.rho_ref;
  const double eta = 3.0 * (p_eos(c, rho) + 0.5 * c.G2 * rho * rho) - rho;
  const double r_ = delta / 19.0, e_ = (-11.0 * delta + 19.0 * eta) / 2394.0, p_ = (3.0 * delta + c.beta2 * eta) / 252.0;
  double o[Q];
  o[0] = r_ - 30.0 * e_ + 12.0 * p_;
  const double ax = r_ - 11.0 * e_ - 4.0 * p_, ce = r_ + 8.0 * e_ + p_;
  for (int i = 1; i < 7; ++i) o[i] = ax;
  for (int i = 7; i < Q; ++i) o[i] = ce;
  for (int i = 0; i < Q; ++i) f[size_t(i) * N + n] = T(o[i]);
}

// rho = sum_i fbar_i + rho_ref into an FP64 array.
template <typename T>
__global__ void k_d3_rho(const T* __restrict__ f, double* __restrict__ rho, int N, double rho_ref) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  double a = 0.0;
  for (int i = 0; i < Q; ++i) a += double(f[size_t(i) * N + n]);
  rho[n] = a + rho_ref;
}

// rho u = sum_i e_i fbar_i - F/2 with F = G^2 rho sum_i omega_i rho(x + e_i) e_i.
template <typename T>
__global__ void k_d3_vel(const T* __restrict__ f, const double* __restrict__ rho, double* ux, double* uy, double* uz,
                         int nx, int ny, int nz, double G2) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  const int N = nx * ny * nz;
  if (n >= N) return;
  const int x = n % nx, y = (n / nx) % ny, z = n / (nx * ny);
  double s[3] = {0.0, 0.0, 0.0}, j[3] = {0.0, 0.0, 0.0};
  for (int i = 1; i < Q; ++i) {
    const int xx = wrap(x + cEX[i], nx), yy = wrap(y + cEY[i], ny), zz = wrap(z + cEZ[i], nz);
    const double w = (cEX[i] * cEX[i] + cEY[i] * cEY[i] + cEZ[i] * cEZ[i]) == 1 ? 1.0 / 6.0 : 1.0 / 12.0;
    const double r = rho[(zz * ny + yy) * nx + xx];
    s[0] += w * r * cEX[i];
    s[1] += w * r * cEY[i];
    s[2] += w * r * cEZ[i];
    const double v = double(f[size_t(i) * N + n]);
    j[0] += cEX[i] * v;
    j[1] += cEY[i] * v;
    j[2] += cEZ[i] * v;
  }
  const double r0 = rho[n];
  if (ux) ux[n] = (j[0] - 0.5 * G2 * r0 * s[0]) / r0;
  if (uy) uy[n] = (j[1] - 0.5 * G2 * r0 * s[1]) / r0;
  if (uz) uz[n] = (j[2] - 0.5 * G2 * r0 * s[2]) / r0;
}

// FP64 diagnostics, first stage: block b sums nodes b, b + G, ... in a fixed order
// and writes kReduceSlots3 values: mass, the three components of sum_i e_i fbar_i,
// the number of nodes with rho above `mid`, min rho, max rho, the number of nodes
// whose density is not finite.  Second stage: k_d3_reduce_final (one block).
constexpr int kReduceBlocks3 = 512, kReduceSlots3 = 8;

template <typename T>
__global__ void __launch_bounds__(256) k_d3_reduce_partial(const T* __restrict__ f, int N, double rho_ref, double mid,
                                                            double* __restrict__ part) {
  __shared__ double sh[kReduceSlots3][256];
  double a[kReduceSlots3] = {0.0, 0.0, 0.0, 0.0, 0.0, INFINITY, -INFINITY, 0.0};
  for (int n = blockIdx.x * blockDim.x + threadIdx.x; n < N; n += gridDim.x * blockDim.x) {
    double r = 0.0, jx = 0.0, jy = 0.0, jz = 0.0;
    for (int i = 0; i < Q; ++i) {
      const double v = double(f[size_t(i) * N + n]);
      r += v;
      jx += cEX[i] * v;
      jy += cEY[i] * v;
      jz += cEZ[i] * v;
    }
    r += rho_ref;
    if (!isfinite(r)) {
      a[7] += 1.0;
      continue;
    }
    a[0] += r;
    a[1] += jx;
    a[2] += jy;
    a[3] += jz;
    a[4] += r > mid ? 1.0 : 0.0;
    a[5] = fmin(a[5], r);
    a[6] = fmax(a[6], r);
  }
  for (int k = 0; k < kReduceSlots3; ++k) sh[k][threadIdx.x] = a[k];
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w)
      for (int k = 0; k < kReduceSlots3; ++k) {
        const double x = sh[k][threadIdx.x], y = sh[k][threadIdx.x + w];
        sh[k][threadIdx.x] = k == 5 ? fmin(x, y) : (k == 6 ? fmax(x, y) : x + y);
      }
    __syncthreads();
  }
  if (threadIdx.x < kReduceSlots3) part[blockIdx.x * kReduceSlots3 + threadIdx.x] = sh[threadIdx.x][0];
}

// (One warp per slot, lanes over the blocks, a fixed order.)
__global__ void __launch_bounds__(32 * kReduceSlots3)
    k_d3_reduce_final(const double* __restrict__ part, int blocks, double* __restrict__ out) {
  const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double a = k == 5 ? INFINITY : (k == 6 ? -INFINITY : 0.0);
  auto fold = [&](double x, double y) { return k == 5 ? fmin(x, y) : (k == 6 ? fmax(x, y) : x + y); };
  for (int b = lane; b < blocks; b += 32) a = fold(a, part[b * kReduceSlots3 + k]);
  for (int w = 16; w > 0; w >>= 1) a = fold(a, __shfl_xor_sync(0xffffffffu, a, w));
  if (lane == 0) out[k] = a;
}

}  // namespace

struct lb_d3_handle {
  lb_params p;
  lb_derived d;
  int nz;
  void* f[2];
  int cur;
  bool overlap;  // the steps' launches may overlap their predecessor's end (lbm_launch.cuh)
  cudaStream_t stream;
  CV3<r64> c64;
  CV3<f2> c32;
  C3<float> cpull;  // of k_d3_pull
  bool vec;         // rows of a multiple of 16 bytes (and both buffers aligned)
  bool windows;     // k_d3_step (else k_d3_pull)
  bool can_window, can_pull, auto_windows;  // forms that the lattice allows, and the one by rule
  int sms;
  bool have_maps;   // tensor maps of both buffers
  CUtensorMap maps[2];
  int* wait_error;  // device word set by a bounded wait that gave up (behind `part`)
  int tw, th, tz;  // tile of the step kernel and planes of its z-chunks
  // Graphs of kD3GraphSteps steps starting from buffer 0 and 1 (captured on first
  // use on the handle's private stream, launched on `stream`); graph_failed: a
  // capture failed once, so plain launches are used from then on.
  cudaStream_t cstream = nullptr;
  cudaGraph_t graph[2] = {nullptr, nullptr};
  cudaGraphExec_t exec[2] = {nullptr, nullptr};
  bool graph_failed = false;
  double* part = nullptr;  // reduction partials (kReduceBlocks3 x kReduceSlots3) and the result
  char err[512];
};

namespace {

using namespace lbm;

int fail3(lb_d3_handle* h, int code, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  std::vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  if (h)
    std::snprintf(h->err, sizeof(h->err), "%s", buf);
  else
    set_thread_error(buf);
  return code;
}

size_t nodes(const lb_params* p, int nz) { return size_t(p->nx) * size_t(p->ny) * size_t(nz); }

// 3-D parameters: the thermodynamics of lb_derive (Eqs. 17-22 hold unchanged),
// the 3-D coefficients of Eq. 7 and the 3-D closure of Eq. 16.
int derive3(const lb_params* p, int nz, lb_derived* d, char* err, size_t n) {
  auto bad = [&](int code, const char* m) {
    std::snprintf(err, n, "%s", m);
    return code;
  };
  if (!p || !d) return bad(LB_EINVAL, "null argument");
  if (p->nx < 1 || p->ny < 1 || nz < 1) return bad(LB_EINVAL, "nx, ny and nz must be >= 1");
  if (int64_t(p->nx) * p->ny * nz >= (int64_t(1) << 31))
    return bad(LB_EINVAL, "lattice too large: nx ny nz must be below 2^31");
  if (p->precision == LB_FP16S) return bad(LB_ENOTSUP, "the D3Q19 step stores FP64 or FP32 populations");
  if (p->layout != LB_LAYOUT_PLANES) return bad(LB_ENOTSUP, "the D3Q19 step uses the planes layout");
  if (p->variant != LB_AUTO && p->variant != LB_FUSED) return bad(LB_ENOTSUP, "the D3Q19 step is the fused one");
  const double w = p->varpi == 0.0 ? 1.0 / 6.0 : p->varpi;
  if (!(w > 0) || w == 1.0 || std::fabs(w - 7.0 / 18.0) < 1e-12)
    return bad(LB_EINVAL, "varpi must be > 0 and not 1 or 7/18 (singular 3-D coefficients)");
  lb_params q = *p;
  q.nx = q.nx < 3 ? 3 : q.nx;
  q.ny = q.ny < 3 ? 3 : q.ny;
  q.varpi = 1.0 / 6.0;  // validated above; the 2-D coefficients are replaced below
  q.s_q = q.s_e = q.s_eps = 1.0;
  const int rc = derive(&q, d, err, n);
  if (rc != LB_OK) return rc;
  const double k = 38.0 * (1.0 - w) / 11.0;
  d->k = k;
  d->beta2 = -19.0 / k;
  d->b = 21.0 * (1.0 - w) / (5.0 * (7.0 - 18.0 * w));
  d->h = 798.0 * w * (1.0 - w) / (5.0 * (7.0 - 18.0 * w));
  const double tau_p = 1.0 / p->s_p - 0.5;
  const double tau_q = 1.0 / (12.0 * tau_p);
  const double tau_e = 1.0 / (12.0 * (1.0 + 5.0 * k / 19.0) * tau_q);
  d->s_q = p->s_q > 0 ? p->s_q : 1.0 / (tau_q + 0.5);
  d->s_e = p->s_e > 0 ? p->s_e : 1.0 / (tau_e + 0.5);
  d->s_eps = p->s_eps > 0 ? p->s_eps : kSEps3;
  auto ok = [](double s) { return s > 0.0 && s < 2.0; };
  if (!ok(d->s_q) || !ok(d->s_e) || !ok(d->s_eps)) return bad(LB_EINVAL, "relaxation rates must lie in (0, 2)");
  return LB_OK;
}

template <typename T>
C3<T> make_c3(const lb_params& p, const lb_derived& d) {
  C3<T> c;
  c.eos = p.eos;
  c.rho_ref = T(p.rho_ref);
  c.G2 = T(d.G2);
  c.lam_RT = T(d.lam * p.R_gas * d.T);
  c.lam_a = T(d.lam * p.eos_a);
  c.b = T(p.eos_b);
  c.bq = T(p.eos_b / 4.0);
  c.se = T(d.s_e);
  c.seps = T(d.s_eps);
  c.sq = T(d.s_q);
  c.sp = T(d.s_p);
  c.sm = T(d.s_q);
  c.spi = T(d.s_eps);
  c.k_seps_ome = T(d.k * d.s_eps * (d.s_e / 2.0 - 1.0));
  c.h_sq_ome = T(d.h * d.s_q * (d.s_e / 2.0 - 1.0));
  c.b_sq_omp = T(d.b * d.s_q * (d.s_p / 2.0 - 1.0));
  c.beta2 = T(d.beta2);
  return c;
}

template <typename V>
CV3<V> make_cv3(const lb_params& p, const lb_derived& d) {
  auto m = [](double v) { return Val<V>::make(v); };
  const double om_e = d.s_e / 2.0 - 1.0, om_p = d.s_p / 2.0 - 1.0;
  const double bq = d.b * d.s_q * om_p, s_m = d.s_q, s_pi = d.s_eps;
  const double RT = p.R_gas * d.T, cA = 1.5 * d.G2 - 3.0 * d.lam * p.eos_a;
  CV3<V> c;
  c.eos = p.eos;
  c.rho_ref = m(p.rho_ref);
  c.nbq = m(p.eos == LB_EOS_VDW ? -p.eos_b : -p.eos_b / 4.0);
  c.lam_RT3 = m(3.0 * d.lam * RT);
  c.cA = m(cA);
  c.G2s = m(d.G2 / 12.0);
  c.gq = m(d.G2 / 1728.0);
  c.lam_RT3_lo = Val<V>::low(3.0 * d.lam * RT);
  c.cA_lo = Val<V>::low(cA);
  c.G2s_lo = Val<V>::low(d.G2 / 12.0);
  c.se = m(d.s_e);
  c.kse = m(d.k * d.s_eps * om_e / 19.0);
  c.hq = m(d.h * d.s_q * om_e * 5.0 / 57.0);
  c.ceta = m(-(d.beta2 + 5.5));
  c.seps_a = m(d.s_eps / 10.5);
  c.sp3 = m(d.s_p / 3.0);
  c.spi3 = m(s_pi / 3.0);
  c.bq2 = m(bq * 10.0 / 3.0);
  c.bq23 = m(bq * 10.0 / 9.0);
  c.nbq23 = m(-bq * 10.0 / 9.0);
  c.nsp = m(-d.s_p);
  c.nbq5 = m(-bq * 5.0 / 3.0);
  c.sq6 = m(d.s_q / 6.0);
  c.om8 = m((1.0 - s_m) / 8.0);
  c.one = m(1.0);
  c.two = m(2.0);
  c.three = m(3.0);
  c.half = m(0.5);
  c.quarter = m(0.25);
  c.nquarter = m(-0.25);
  c.eighth = m(0.125);
  c.n2 = m(-2.0);
  c.n3 = m(-3.0);
  c.n4 = m(-4.0);
  c.nhalf = m(-0.5);
  c.nthird = m(-1.0 / 3.0);
  c.sixth = m(1.0 / 6.0);
  c.n12 = m(-1.0 / 12.0);
  c.i24 = m(1.0 / 24.0);
  c.n2h = m(-2.5);
  c.n5h = m(-5.5);
  c.n10h = m(-10.5);
  c.c1375 = m(13.75);
  c.c1121 = m(11.0 / 21.0);
  return c;
}

// Planes per z-chunk (at most `most`) of a lattice of xy tiles, and the time of a step in
// planes of a block.  A block costs its planes and `extra` more (the two planes whose
// densities alone it needs).  The blocks start in order as places fall free: whole
// rounds of the full chunks, then the chunks of the remainder, which go first into the
// places that the last round leaves.  64^3 FP32 (us a step): 4 planes 14.1, 3 planes
// 17.9; 96^3: 12 planes 33.4, 6 planes 37.3; 128^3: 14 planes 74.9, 16 planes 79.8.
// (FP32 windows: at most 32 planes and 1.2 more.)
constexpr int kWindowPlanes = 32;
constexpr double kWindowExtra = 1.2;
double chunk_planes(long long xy, int nz, int places, int most, double extra, int* tz_out) {
  double best_cost = 1e300;
  for (int tz = 1; tz <= nz && tz <= most; ++tz) {
    const long long full = xy * (nz / tz), rounds = full / places, over = full % places;
    const int rem = nz % tz;
    const double d1 = tz + extra, d2 = rem + extra;
    double cost = double(rounds + (over ? 1 : 0)) * d1;
    if (rem) {
      const long long room = over ? (places - over) * (long long)(d1 / d2) : 0;
      if (xy > room) cost += double((xy - room + places - 1) / places) * d2;
    }
    if (cost < best_cost) {
      best_cost = cost;
      *tz_out = tz;
    }
  }
  return best_cost;
}

// Tile and chunk of the step.  FP32: 32 x 8 tiles.  FP64: the FP64 pipe bounds the step, a
// plane of a block takes as long as its schedulers' largest number of warps, and the SM
// with the most planes ends last; so the tile of at most 256 nodes (even width, for the
// 16-byte copies) and the chunk with the least time are taken: 120 x 100 x 71 in chunks of
// 10 x 25 x 23 nodes, 539 us a step, against 607 with 32 x 8 x 5; 33 x 77 x 50 in chunks
// of 12 x 10 x 8, 104 us against 168.
template <typename T>
void tile_plan(lb_d3_handle* h, int sms) {
  using W = Win3<T>;
  const int nx = h->p.nx, ny = h->p.ny, nz = h->nz;
  auto tiles = [&](int tw, int th) { return (long long)((nx + tw - 1) / tw) * ((ny + th - 1) / th); };
  h->tw = TX;
  h->th = TY;
  if (W::fixed) {
    chunk_planes(tiles(TX, TY), nz, sms * d3_blocks<T>(), kWindowPlanes, kWindowExtra, &h->tz);
    return;
  }
  double best = 1e300;
  for (int tw = 8; tw <= 64; tw += 2)
    for (int th = 4; th * tw <= W::threads && th <= 32; ++th) {
      if ((th + 2) * (tw + 2 * W::run) > W::cells || (th + 2) * (tw + 2 * W::run) / W::run > W::threads) continue;
      if ((th + 2) * (tw + 2) > W::ring_cells || 2 * (tw + 2) + 2 * th > W::threads) continue;
      // Warps a scheduler works off per plane: nodes, and 18 of about 300 instructions for the ring.
      const double plane = (tw * th + 127) / 128 + 0.06 * ((2 * (tw + 2) + 2 * th + 127) / 128);
      if (plane * double(tiles(tw, th)) * nz / (sms * d3_blocks<T>()) >= best) continue;  // even if spread evenly
      int tz = 1;
      const double cost = plane * chunk_planes(tiles(tw, th), nz, sms * d3_blocks<T>(), nz, 0.4, &tz);
      if (cost < best * 0.999) {
        best = cost;
        h->tw = tw;
        h->th = th;
        h->tz = tz;
      }
    }
}

// k_d3_pull: 32 planes (fewest halo planes) unless that leaves fewer than two waves of
// resident blocks (3 per SM); then halved down to 2.
int chunk_planes_pull(int nx, int ny, int nz, int sms) {
  const long long xy = (long long)((nx + TX - 1) / TX) * ((ny + kPullTY - 1) / kPullTY);
  int tz = kPullTZ;
  while (tz > 2 && xy * ((nz + tz - 1) / tz) < 2LL * 3 * sms) tz /= 2;
  return tz;
}

// Whether an FP32 lattice steps faster by windows (k_d3_step) than by pulls (k_d3_pull), from
// the planes that the last SM to finish works off.  Windows: chunk_planes.  Pulls: rounds of
// 3 blocks per SM of tz planes and 2.5 more, the last one by half its fill and half whole; a
// plane of a block of pulls costs more in the company of later rounds (sqrt(rounds)), and
// windows lose what their 32 x 8 tiles hold outside the lattice.  The constant is from 159
// lattices of 24 to 256 nodes a side, both forms timed on each: the form taken is the faster
// or within 2% of it on 140, within 9% on all but two (120 x 124 x 33: 25.8 us, pulls 22.8;
// 240 x 160 x 48: 76.0, windows 67.8).
// Without the estimate, windows wherever the rows filled their tiles: 40^3 10.2 us a step
// against 6.3 by pulls, 40 x 72 x 101 23.4 / 18.5, 104^3 57.0 / 50.2, 120 x 40 x 40 12.4 / 11.8, and
// pulls at 196 x 35 x 48 21.2 / 19.1; windows are taken at 64^3 14.1 / 15.2, 96^3 33.9 / 41.2,
// 160^3 133 / 152, 256^3 461 / 526.
bool windows_win(int nx, int ny, int nz, int sms) {
  const long long xy = (long long)((nx + TX - 1) / TX) * ((ny + TY - 1) / TY);
  int tz = 1;
  const double windows = chunk_planes(xy, nz, sms * d3_blocks<float>(), kWindowPlanes, kWindowExtra, &tz);
  tz = chunk_planes_pull(nx, ny, nz, sms);
  const long long places = 3LL * sms;
  const long long blocks =
      (long long)((nx + TX - 1) / TX) * ((ny + kPullTY - 1) / kPullTY) * ((nz + tz - 1) / tz);
  const long long rounds = (blocks + places - 1) / places;
  const double last = double(blocks - places * (rounds - 1)) / double(places);
  const double pulls = (double(rounds) - 0.5 + 0.5 * last) * (tz + 2.5);
  const double fill = double(nx) * ny / (double(xy) * TX * TY);
  return windows < 0.37 * pulls * fill * std::sqrt(double(rounds));
}

// The step's windows by tensor copies where possible (FP32), else by 16-byte copies; FP32
// rows that are no multiple of 16 bytes or shorter than a window (24 x 31 x 200: 11.5 us a step
// against 13.3) take k_d3_pull.
template <typename T>
cudaError_t configure_step(lb_d3_handle* h, int sms) {
  h->vec = (size_t(h->p.nx) * sizeof(T)) % 16 == 0 && reinterpret_cast<uintptr_t>(h->f[0]) % 16 == 0 &&
           reinterpret_cast<uintptr_t>(h->f[1]) % 16 == 0;
  h->can_window = sizeof(T) == 8 || (h->vec && h->p.nx >= Win3<T>::cols);
  h->can_pull = sizeof(T) == 4;
  h->auto_windows = h->can_window && (!h->can_pull || windows_win(h->p.nx, h->p.ny, h->nz, sms));
  h->have_maps = false;
  std::memset(h->maps, 0, sizeof(h->maps));
  using W = Win3<T>;
  if (W::tensor && h->can_window && h->p.ny >= W::rows) {
    h->have_maps = true;
    for (int k = 0; k < 2; ++k)
      h->have_maps = h->have_maps &&
                     encode_volume_map(&h->maps[k], h->f[k], h->p.nx, h->p.ny, h->nz, Q, W::cols, W::rows);
  }
  cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void*>(k_d3_step<T, true>),
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, int(Win3<T>::smem));
  if (e == cudaSuccess && sizeof(T) == 8)
    e = cudaFuncSetAttribute(reinterpret_cast<const void*>(k_d3_step<T, sizeof(T) != 8>),
                             cudaFuncAttributeMaxDynamicSharedMemorySize, int(Win3<T>::smem));
  return e;
}

void take_form(lb_d3_handle* h, bool windows) {
  h->windows = windows;
  if (!windows)
    h->tz = chunk_planes_pull(h->p.nx, h->p.ny, h->nz, h->sms);
  else if (h->p.precision == LB_FP64)
    tile_plan<double>(h, h->sms);
  else
    tile_plan<float>(h, h->sms);
}

void drop_graphs(lb_d3_handle* h) {
  for (int c = 0; c < 2; ++c) {
    if (h->exec[c]) cudaGraphExecDestroy(h->exec[c]);
    if (h->graph[c]) cudaGraphDestroy(h->graph[c]);
    h->exec[c] = nullptr;
    h->graph[c] = nullptr;
  }
}

template <typename T, bool VEC>
void launch_windows(lb_d3_handle* h, const CV3<typename ValOf<T>::V>& c) {
  const lb_params& p = h->p;
  const dim3 grid((p.nx + h->tw - 1) / h->tw, (p.ny + h->th - 1) / h->th, (h->nz + h->tz - 1) / h->tz);
  lbm::launch_step_kernel(
      h->overlap, k_d3_step<T, VEC>, grid, Win3<T>::threads, Win3<T>::smem, h->stream, static_cast<const T*>(h->f[h->cur]), static_cast<T*>(h->f[1 - h->cur]), p.nx, p.ny, h->nz, h->tw,
      h->th, h->tz, c, h->maps[h->cur], h->have_maps ? 1 : 0, h->wait_error);
}

void launch_step(lb_d3_handle* h) {
  const lb_params& p = h->p;
  if (p.precision == LB_FP64) {
    if (h->vec)
      launch_windows<double, true>(h, h->c64);
    else
      launch_windows<double, false>(h, h->c64);
  } else if (h->windows) {
    launch_windows<float, true>(h, h->c32);
  } else {
    const dim3 grid((p.nx + TX - 1) / TX, (p.ny + kPullTY - 1) / kPullTY, (h->nz + h->tz - 1) / h->tz);
    const float* in = static_cast<const float*>(h->f[h->cur]);
    float* out = static_cast<float*>(h->f[1 - h->cur]);
    // 32-bit plane offsets while 19 nx ny nz < 2^31, 64-bit above.
    if (int64_t(Q) * p.nx * p.ny * h->nz >= (int64_t(1) << 31))
      lbm::launch_step_kernel(h->overlap, k_d3_pull<long long>, grid, dim3(TX, kPullTY), 0, h->stream, in, out, p.nx, p.ny, h->nz, h->tz, h->cpull);
    else
      lbm::launch_step_kernel(h->overlap, k_d3_pull<int>, grid, dim3(TX, kPullTY), 0, h->stream, in, out, p.nx, p.ny, h->nz, h->tz, h->cpull);
  }
  h->cur = 1 - h->cur;
}

constexpr int64_t kD3GraphSteps = 64;
static_assert(kD3GraphSteps % 2 == 0, "a graph must end in the buffer it starts from");

// Captures (once) the graph of kD3GraphSteps steps that starts from buffer h->cur.
// Returns false, and leaves plain launches in use, if the capture fails.
bool ensure_graph(lb_d3_handle* h) {
  const int c = h->cur;
  if (h->exec[c]) return true;
  if (h->graph_failed) return false;
  bool ok = h->cstream || cudaStreamCreateWithFlags(&h->cstream, cudaStreamNonBlocking) == cudaSuccess;
  if (ok) ok = cudaStreamBeginCapture(h->cstream, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
  if (ok) {
    cudaStream_t keep = h->stream;
    h->stream = h->cstream;
    for (int64_t k = 0; k < kD3GraphSteps; ++k) launch_step(h);
    h->stream = keep;
    ok = cudaStreamEndCapture(h->cstream, &h->graph[c]) == cudaSuccess && h->graph[c];
    if (ok) ok = cudaGraphInstantiate(&h->exec[c], h->graph[c], 0) == cudaSuccess;
  }
  h->cur = c;  // the captured launches flipped it an even number of times
  if (!ok) {
    cudaGetLastError();
    h->graph_failed = true;
  }
  return ok;
}

}  // namespace

extern "C" {

void lb_d3_velocities(int* ex, int* ey, int* ez) {
  for (int i = 0; i < Q; ++i) {
    if (ex) ex[i] = kEX[i];
    if (ey) ey[i] = kEY[i];
    if (ez) ez[i] = kEZ[i];
  }
}

int lb_d3_derive(const lb_params* p, int32_t nz, lb_derived* out) {
  char err[256];
  lb_derived d;
  const int rc = derive3(p, nz, &d, err, sizeof(err));
  if (rc != LB_OK) return fail3(nullptr, rc, "%s", err);
  if (!out) return fail3(nullptr, LB_EINVAL, "null output");
  *out = d;
  return LB_OK;
}

size_t lb_d3_state_bytes(const lb_params* p, int32_t nz) {
  if (!p || nz < 1) return 0;
  return Q * nodes(p, nz) * (p->precision == LB_FP64 ? 8 : 4);
}

int lb_d3_init(lb_d3_handle** out, const lb_params* p, int32_t nz, void* f_a, void* f_b, const double* rho0,
               int rho0_on_device, void* stream) {
  if (!out) return fail3(nullptr, LB_EINVAL, "null handle pointer");
  *out = nullptr;
  char err[256];
  lb_derived d;
  int rc = derive3(p, nz, &d, err, sizeof(err));
  if (rc != LB_OK) return fail3(nullptr, rc, "%s", err);
  if (!f_a || !f_b || f_a == f_b) return fail3(nullptr, LB_EINVAL, "f_a and f_b must be two distinct device buffers");
  if (!rho0) return fail3(nullptr, LB_EINVAL, "null initial density");
  const size_t N = nodes(p, nz);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  auto cuda_fail = [&](cudaError_t e, const char* what) {
    return fail3(nullptr, LB_ECUDA, "%s: %s", what, cudaGetErrorString(e));
  };
  lb_params q = *p;
  const double* rho_dev = rho0;
  if (!rho0_on_device) {
    cudaError_t e = cudaMemcpyAsync(f_b, rho0, N * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return cuda_fail(e, "copy of the initial density");
    rho_dev = static_cast<const double*>(f_b);
  }
  if (std::isnan(q.rho_ref)) {
    std::vector<double> host;
    const double* hp = rho0;
    if (rho0_on_device) {
      host.resize(N);
      cudaError_t e = cudaMemcpyAsync(host.data(), rho0, N * sizeof(double), cudaMemcpyDeviceToHost, s);
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
      if (e != cudaSuccess) return cuda_fail(e, "read of the initial density");
      hp = host.data();
    }
    double sum = 0.0;
    for (size_t n = 0; n < N; ++n) sum += hp[n];
    q.rho_ref = sum / double(N);
  }
  if (q.precision == LB_FP32) q.rho_ref = double(float(q.rho_ref));
  unsigned long long* bad = nullptr;
  cudaError_t e = cudaMalloc(&bad, 2 * sizeof(unsigned long long));
  if (e != cudaSuccess) return cuda_fail(e, "cudaMalloc of the status words");
  e = cudaMemsetAsync(bad, 0xff, 2 * sizeof(unsigned long long), s);
  const C3<double> c = make_c3<double>(q, d);
  const int threads = 256, blocks = int((N + threads - 1) / threads);
  if (e == cudaSuccess) {
    if (q.precision == LB_FP64)
      k_d3_init<double><<<blocks, threads, 0, s>>>(rho_dev, static_cast<double*>(f_a), int(N), c, bad);
    else
      k_d3_init<float><<<blocks, threads, 0, s>>>(rho_dev, static_cast<float*>(f_a), int(N), c, bad);
    e = cudaGetLastError();
  }
  unsigned long long first[2] = {~0ull, ~0ull};
  if (e == cudaSuccess) e = cudaMemcpyAsync(first, bad, sizeof(first), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(bad);
  if (e != cudaSuccess) return cuda_fail(e, "initial state");
  if (first[0] != ~0ull)
    return fail3(nullptr, LB_EINVAL, "initial density at node %llu is not positive and finite", first[0]);
  if (first[1] != ~0ull) return fail3(nullptr, LB_EINVAL, "initial density at node %llu exceeds 1/b of the vdW EOS", first[1]);
  lb_d3_handle* h = new (std::nothrow) lb_d3_handle();
  if (!h) return fail3(nullptr, LB_EINVAL, "out of host memory");
  h->p = q;
  h->d = d;
  h->nz = nz;
  h->f[0] = f_a;
  h->f[1] = f_b;
  h->cur = 0;
  h->stream = s;
  h->c64 = make_cv3<r64>(q, d);
  h->c32 = make_cv3<f2>(q, d);
  h->cpull = make_c3<float>(q, d);
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    sms = 152;
  }
  h->err[0] = 0;
  auto give_up = [&](cudaError_t ce, const char* what) {
    cudaGetLastError();
    delete h;
    return cuda_fail(ce, what);
  };
  e = q.precision == LB_FP64 ? configure_step<double>(h, sms) : configure_step<float>(h, sms);
  if (e != cudaSuccess) return give_up(e, "step configuration");
  h->sms = sms;
  take_form(h, h->auto_windows);
  if (cudaMalloc(&h->part, (kReduceBlocks3 + 2) * kReduceSlots3 * sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    delete h;
    return fail3(nullptr, LB_ENOMEM, "cudaMalloc of the %zu-byte reduction workspace",
                 size_t(kReduceBlocks3 + 2) * kReduceSlots3 * sizeof(double));
  }
  h->wait_error = reinterpret_cast<int*>(h->part + (kReduceBlocks3 + 1) * kReduceSlots3);
  e = cudaMemsetAsync(h->wait_error, 0, sizeof(int), s);
  if (e != cudaSuccess) {
    cudaFree(h->part);
    return give_up(e, "cudaMemsetAsync of the wait word");
  }
  *out = h;
  return LB_OK;
}

int lb_d3_step(lb_d3_handle* h, int64_t nsteps) {
  if (!h) return fail3(nullptr, LB_EINVAL, "null handle");
  if (nsteps < 0) return fail3(h, LB_EINVAL, "nsteps must be >= 0");
  // Runs of kD3GraphSteps steps replay a graph, unless the caller's stream is being
  // captured itself (then the steps go into the caller's graph as plain launches).
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  if (h->stream != nullptr && cudaStreamIsCapturing(h->stream, &capture) != cudaSuccess) {
    cudaGetLastError();
    capture = cudaStreamCaptureStatusActive;
  }
  h->overlap = capture == cudaStreamCaptureStatusNone;
  while (capture == cudaStreamCaptureStatusNone && nsteps >= kD3GraphSteps && ensure_graph(h)) {
    const cudaError_t e = cudaGraphLaunch(h->exec[h->cur], h->stream);
    if (e != cudaSuccess) return fail3(h, LB_ECUDA, "step graph launch: %s", cudaGetErrorString(e));
    nsteps -= kD3GraphSteps;  // an even number of steps: the state is back in the same buffer
  }
  for (int64_t k = 0; k < nsteps; ++k) launch_step(h);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail3(h, LB_ECUDA, "step launch: %s", cudaGetErrorString(e));
  return LB_OK;
}

int lb_d3_moments(lb_d3_handle* h, void* rho, void* ux, void* uy, void* uz) {
  if (!h) return fail3(nullptr, LB_EINVAL, "null handle");
  if (!rho) return fail3(h, LB_EINVAL, "rho output is required");
  const int N = int(nodes(&h->p, h->nz));
  const int threads = 256, blocks = (N + threads - 1) / threads;
  double* r = static_cast<double*>(rho);
  const void* f = h->f[h->cur];
  if (h->p.precision == LB_FP64)
    k_d3_rho<double><<<blocks, threads, 0, h->stream>>>(static_cast<const double*>(f), r, N, h->p.rho_ref);
  else
    k_d3_rho<float><<<blocks, threads, 0, h->stream>>>(static_cast<const float*>(f), r, N, h->p.rho_ref);
  if (ux || uy || uz) {
    double *a = static_cast<double*>(ux), *b = static_cast<double*>(uy), *c = static_cast<double*>(uz);
    if (h->p.precision == LB_FP64)
      k_d3_vel<double><<<blocks, threads, 0, h->stream>>>(static_cast<const double*>(f), r, a, b, c, h->p.nx, h->p.ny,
                                                          h->nz, h->d.G2);
    else
      k_d3_vel<float><<<blocks, threads, 0, h->stream>>>(static_cast<const float*>(f), r, a, b, c, h->p.nx, h->p.ny,
                                                         h->nz, h->d.G2);
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail3(h, LB_ECUDA, "moments launch: %s", cudaGetErrorString(e));
  return LB_OK;
}

int lb_d3_reduce(lb_d3_handle* h, double out[8]) {
  if (!h) return fail3(nullptr, LB_EINVAL, "null handle");
  if (!out) return fail3(h, LB_EINVAL, "null output");
  const int N = int(nodes(&h->p, h->nz));
  const double mid = 0.5 * (h->d.rho_g + h->d.rho_l);
  const int blocks = std::min(kReduceBlocks3, (N + 255) / 256);
  const void* f = h->f[h->cur];
  if (h->p.precision == LB_FP64)
    k_d3_reduce_partial<double><<<blocks, 256, 0, h->stream>>>(static_cast<const double*>(f), N, h->p.rho_ref, mid,
                                                                h->part);
  else
    k_d3_reduce_partial<float><<<blocks, 256, 0, h->stream>>>(static_cast<const float*>(f), N, h->p.rho_ref, mid,
                                                               h->part);
  double* res = h->part + kReduceBlocks3 * kReduceSlots3;
  k_d3_reduce_final<<<1, 32 * kReduceSlots3, 0, h->stream>>>(h->part, blocks, res);
  cudaError_t e = cudaMemcpyAsync(out, res, kReduceSlots3 * sizeof(double), cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return fail3(h, LB_ECUDA, "reduction: %s", cudaGetErrorString(e));
  if (out[7] > 0) return fail3(h, LB_ENONFINITE, "%.0f nodes have a non-finite density", out[7]);
  return LB_OK;
}

int lb_d3_form(const lb_d3_handle* h) { return !h ? LB_EINVAL : h->windows ? LB_D3_WINDOWS : LB_D3_PULLS; }

int lb_d3_set_form(lb_d3_handle* h, int form) {
  if (!h) return fail3(nullptr, LB_EINVAL, "null handle");
  if (form != LB_D3_AUTO && form != LB_D3_PULLS && form != LB_D3_WINDOWS)
    return fail3(h, LB_EINVAL, "form must be LB_D3_AUTO, LB_D3_PULLS or LB_D3_WINDOWS");
  if ((form == LB_D3_PULLS && !h->can_pull) || (form == LB_D3_WINDOWS && !h->can_window))
    return fail3(h, LB_ENOTSUP, "the lattice does not step in this form");
  const bool windows = form == LB_D3_AUTO ? h->auto_windows : form == LB_D3_WINDOWS;
  if (windows == h->windows) return LB_OK;
  drop_graphs(h);  // captured with the other form
  take_form(h, windows);
  return LB_OK;
}

int lb_d3_status(lb_d3_handle* h) {
  if (!h) return fail3(nullptr, LB_EINVAL, "null handle");
  int v = 0;
  cudaError_t e = cudaMemcpyAsync(&v, h->wait_error, sizeof(int), cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  if (e == cudaSuccess && v) e = cudaMemsetAsync(h->wait_error, 0, sizeof(int), h->stream);
  if (e != cudaSuccess) return fail3(h, LB_ECUDA, "status: %s", cudaGetErrorString(e));
  return v ? fail3(h, LB_ETIMEOUT, "a bounded wait for a tensor copy gave up") : LB_OK;
}

void* lb_d3_state(const lb_d3_handle* h) { return h ? h->f[h->cur] : nullptr; }

int lb_d3_get_state(lb_d3_handle* h, void* dst) {
  if (!h || !dst) return fail3(h, LB_EINVAL, "null argument");
  const cudaError_t e = cudaMemcpyAsync(dst, h->f[h->cur], lb_d3_state_bytes(&h->p, h->nz), cudaMemcpyDeviceToDevice,
                                        h->stream);
  if (e != cudaSuccess) return fail3(h, LB_ECUDA, "state copy: %s", cudaGetErrorString(e));
  return LB_OK;
}

int lb_d3_set_state(lb_d3_handle* h, const void* src) {
  if (!h || !src) return fail3(h, LB_EINVAL, "null argument");
  const cudaError_t e = cudaMemcpyAsync(h->f[h->cur], src, lb_d3_state_bytes(&h->p, h->nz), cudaMemcpyDeviceToDevice,
                                        h->stream);
  if (e != cudaSuccess) return fail3(h, LB_ECUDA, "state copy: %s", cudaGetErrorString(e));
  return LB_OK;
}

int lb_d3_get_params(const lb_d3_handle* h, lb_params* out, lb_derived* derived) {
  if (!h) return fail3(nullptr, LB_EINVAL, "null handle");
  if (out) *out = h->p;
  if (derived) *derived = h->d;
  return LB_OK;
}

const char* lb_d3_last_error(const lb_d3_handle* h) { return h ? h->err : thread_error(); }

void lb_d3_free(lb_d3_handle* h) {
  if (!h) return;
  drop_graphs(h);
  if (h->cstream) cudaStreamDestroy(h->cstream);
  if (h->part) cudaFree(h->part);
  delete h;
}

}  // extern "C"
