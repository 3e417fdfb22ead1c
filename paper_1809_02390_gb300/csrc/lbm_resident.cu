// Host side of the resident run (lbm_resident.cuh): the cut of a lattice into tiles,
// the exchange buffer's size and the cooperative launch.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <mutex>
#include <vector>

#include "lbm_resident.cuh"
#include "lbm_handle.cuh"

namespace lbm {

namespace {

template <typename V, typename S>
constexpr const void* kernel_of() {
  return reinterpret_cast<const void*>(k_resident<V, S>);
}

const void* res_kernel(int precision) {
  switch (precision) {
    case LB_FP64: return kernel_of<double, double>();
    case LB_FP32: return kernel_of<f2, float>();
    default: return kernel_of<f2, __half>();
  }
}

size_t res_smem(int precision, int wmax, int hmax, int pitch) {
  const size_t plane = size_t(pitch) * (hmax + 4);
  const size_t real = precision == LB_FP64 ? 8 : 4, store = precision == LB_FP64 ? 8 : precision == LB_FP32 ? 4 : 2;
  return size_t(res_table_bytes(wmax, hmax, precision == LB_FP64 ? 1 : 2)) + plane * (real + 18 * store);
}

// Steps of one launch (even, so that a full chunk ends where it started): about 5 ms, so that
// other work on the GPU gets its turn, by the plan's cost and some 3000 cycles a step of what
// it leaves out (FP32 256^2 4,300 cycles a step, estimated 4,200; FP64 64^2 15,600 / 18,100;
// FP64 410^2 at 9 rounds of warps 138,000, 72 steps: a fixed number of 4096 held the GPU for
// 9 ms, 31 ms and some 0.3 s).
int res_chunk(double cost) {
  const int n = int(1e7 / (cost + 3000.0)) / 2 * 2;
  return n < 16 ? 16 : n > 4096 ? 4096 : n;
}

}  // namespace

// The cut with the smallest estimated step: a block's warps take the collision in
// turn (FP64: 19 cycles of an SM per warp instruction, four warps at a time; FP32:
// about 130 cycles of an SM per warp of pairs, and no less than the latency of one),
// and each edge node costs its share of the exchange.
bool res_plan(int nx, int ny, int precision, ResPlan* out) {
  const bool fp64 = precision == LB_FP64;
  const int lanes = fp64 ? 1 : 2;
  const int max_threads = fp64 ? ResTraits<double>::max_threads : ResTraits<float>::max_threads;
  double best = 0.0;
  bool found = false;
  for (int gx = 1; gx <= kResTiles && (gx == 1 || nx / gx >= 4); ++gx) {
      int gy = kResTiles / gx;
      if (gy > ny / 4) gy = ny / 4;
      if (gy < 1) gy = 1;
      const int w = (nx + gx - 1) / gx, h = (ny + gy - 1) / gy;
      if (nx / gx < 2 || ny / gy < 2) continue;
      if ((long long)(w + 4) * (h + 4) > 65535) continue;
      // Warps run along the inner rows of w - 4 nodes: with a pitch that is w - 4 modulo
      // the 32 banks, a warp that crosses into the next row stays free of conflicts
      // (512^2 FP32: 4.54 -> 4.34 us a step), where the shared memory allows it.
      int pitch = w > 4 ? w - 4 + (w + 4 - (w - 4) + 31) / 32 * 32 : w + 4;
      if (res_smem(precision, w, h, pitch) > kResSmem - 1024) pitch = w + 4;
      if (res_smem(precision, w, h, pitch) > kResSmem - 1024) continue;
      const int items = res_slots(w, h, lanes).total;
      const int warps = (items + 31) / 32;
      const double work = fp64 ? 15000.0 * ((warps + 3) / 4) : (130.0 * warps > 900.0 ? 130.0 * warps : 900.0);
      const double cost = work + 4.0 * (w + h) + 0.01 * gx * gy;  // cycles
      if (found && cost >= best) continue;
      best = cost;
      found = true;
      const int rounds = (items + max_threads - 1) / max_threads;
      int threads = ((items + rounds - 1) / rounds + 31) / 32 * 32;
      if (threads < 128) threads = 128;
      *out = ResPlan{gx, gy, w, h, pitch, threads, unsigned(res_smem(precision, w, h, pitch)),
                     size_t(gx) * gy * 6 * (w + h) * (fp64 ? 2 : 1), res_chunk(cost)};
    }
  return found;
}

// Most nodes of a resident FP32 or FP16 lattice (res_configure); FP64 lattices of that size
// do not fit the SMs' shared memory.
constexpr long long kResNodes = 340000;

// Largest over the precisions, so that the scratch size differs between them by the
// density plane alone.
size_t res_mail_bytes(int nx, int ny) {
  size_t words = 0;
  if ((long long)nx * ny > kResNodes) return 0;
  for (int precision : {int(LB_FP64), int(LB_FP32), int(LB_FP16S)}) {
    ResPlan p;
    if (res_plan(nx, ny, precision, &p) && p.words > words) words = p.words;
  }
  return 2 * words * sizeof(uint4);
}

namespace {
// Live handles that have made a call long enough to run resident, by device and stream (an
// entry goes with its last handle), and the number of streams per device, which every step
// call reads.
struct Live {
  int dev;
  cudaStream_t stream;
  int handles;
};
constexpr int kDevices = 64;
std::mutex g_live_mu;
std::vector<Live> g_live;
std::atomic<int> g_live_streams[kDevices];

Live* find_live(const lb_handle* h) {
  for (Live& l : g_live)
    if (l.dev == h->res_dev && l.stream == h->stream) return &l;
  return nullptr;
}
}  // namespace

void res_enter(lb_handle* h) {
  if (h->res_live) return;
  std::lock_guard<std::mutex> lock(g_live_mu);
  h->res_live = true;
  if (Live* l = find_live(h)) {
    ++l->handles;
    return;
  }
  g_live.push_back(Live{h->res_dev, h->stream, 1});
  ++g_live_streams[h->res_dev % kDevices];
}

void res_leave(lb_handle* h) {
  if (!h || !h->res_live) return;
  std::lock_guard<std::mutex> lock(g_live_mu);
  for (size_t k = 0; k < g_live.size(); ++k)
    if (g_live[k].dev == h->res_dev && g_live[k].stream == h->stream) {
      if (--g_live[k].handles == 0) {
        g_live.erase(g_live.begin() + k);
        --g_live_streams[h->res_dev % kDevices];
      }
      break;
    }
  h->res_live = false;
}

int res_streams(const lb_handle* h) {
  const std::atomic<int>& streams = g_live_streams[h->res_dev % kDevices];
  if (h->res_live) return streams.load(std::memory_order_relaxed);
  std::lock_guard<std::mutex> lock(g_live_mu);
  return streams.load(std::memory_order_relaxed) + (find_live(h) ? 0 : 1);
}

cudaError_t res_configure(lb_handle* h, void* mail) {
  h->use_res = false;
  h->res_mode = -1;
  h->res_refuse = -1;
  ResPlan p;
  // FP32 and FP16 up to kResNodes: above, a tile's pitch no longer avoids bank conflicts
  // and a step is no faster than a launch of k_step_fused (us: FP32 576^2 4.9 against 5.3,
  // 600^2 6.8 / 5.6; FP16 400^2 3.8 / 3.9, 512^2 5.2 / 4.7, 576^2 6.0 / 6.2, 640 x 600 7.0 / 6.6).
  if (h->p.precision != LB_FP64 && (long long)h->p.nx * h->p.ny > kResNodes) return cudaSuccess;
  if (!mail || h->variant != LB_FUSED || !res_plan(h->p.nx, h->p.ny, h->p.precision, &p)) return cudaSuccess;
  const void* k = res_kernel(h->p.precision);
  int dev = 0, coop = 0, sms = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // The limit is the kernel's, not the handle's: always the largest any plan needs.
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kResSmem - 1024));
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, p.threads, p.smem);
  if (e != cudaSuccess) return e;
  if (!coop || per_sm < 1 || sms < p.gx * p.gy) return cudaSuccess;
  h->res = p;
  h->res_mail = mail;
  h->res_fit = per_sm * sms / (p.gx * p.gy);
  h->res_dev = dev;
  h->use_res = true;
  return cudaSuccess;
}

namespace {

template <typename V, typename S>
cudaError_t launch(lb_handle* h, const VCoef<V>& c, const void* fin, void* fout, void* rec, int rec_first,
                   int rec_every, int nsteps) {
  const ResPlan& p = h->res;
  ResArgs<S> a{static_cast<const S*>(fin),
               static_cast<S*>(fout),
               static_cast<S*>(rec),
               9ll * h->p.nx * h->p.ny,
               rec_first,
               rec_every,
               static_cast<uint4*>(h->res_mail),
               h->wait_error,
               unsigned(h->steps),
               nsteps,
               h->p.nx,
               h->p.ny,
               p.gx,
               p.gy,
               p.wmax,
               p.hmax,
               p.pitch,
               h->p.rounding == LB_ROUND_STOCHASTIC,
               h->st};
  VCoef<V> cc = c;
  void* args[] = {&a, &cc};
  return cudaLaunchCooperativeKernel(kernel_of<V, S>(), dim3(p.gx * p.gy), dim3(p.threads), args, p.smem, h->stream);
}

}  // namespace

// Launches that the device refuses for what else limits the stream (a green context with
// fewer SMs than the device, a debugger's or a partition's limits): single launches still run.
bool res_refused(cudaError_t e) {
  return e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorLaunchOutOfResources || e == cudaErrorNotSupported ||
         e == cudaErrorInvalidConfiguration || e == cudaErrorNotPermitted;
}

// (A launch takes at most 4096 steps, so larger distances are all the same to it.)
static int to_int(int64_t v) { return v > INT32_MAX ? INT32_MAX : int(v); }

cudaError_t res_run(lb_handle* h, int64_t nsteps, void* rec, int64_t every, int64_t* done) {
  int64_t first = every;  // steps until the next recorded state
  *done = 0;
  while (*done < nsteps) {
    // Never a launch of one step: it could not write its result in place.
    const int64_t chunk = h->res.steps, left = nsteps - *done;
    const int64_t n = left <= chunk ? left : (left == chunk + 1 ? chunk - 2 : chunk);
    const void* in = h->f[h->cur];
    void* out = h->f[n & 1 ? 1 - h->cur : h->cur];
    cudaError_t e;
    if (h->res_refuse >= 0 && h->res_refuse-- == 0)
      e = cudaErrorCooperativeLaunchTooLarge;  // lb_resident_selftest
    else
      switch (h->p.precision) {
        case LB_FP64: e = launch<double, double>(h, h->cd, in, out, rec, to_int(first), to_int(every), int(n)); break;
        case LB_FP32: e = launch<f2, float>(h, h->c2, in, out, rec, to_int(first), to_int(every), int(n)); break;
        default: e = launch<f2, __half>(h, h->c2, in, out, rec, to_int(first), to_int(every), int(n)); break;
      }
    if (res_refused(e)) {
      cudaGetLastError();
      h->use_res = false;
      res_leave(h);
      return cudaSuccess;
    }
    if (e != cudaSuccess) return e;
    if (rec) {
      const int64_t states = n >= first ? 1 + (n - first) / every : 0;
      rec = static_cast<char*>(rec) + size_t(states) * lb_state_bytes(&h->p);
      first = states ? every - (n - first) % every : first - n;
    }
    h->steps += n;
    if (n & 1) h->cur = 1 - h->cur;
    *done += n;
  }
  return cudaSuccess;
}

}  // namespace lbm
