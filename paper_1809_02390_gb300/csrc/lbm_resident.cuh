// Many steps of one lattice in a single cooperative launch (sm_103a): the lattice
// is cut into at most one tile per SM, a tile's populations stay in its SM's shared
// memory for all steps, and only the edges travel between SMs.
//
// What bounds short steps: with one launch per step (graph replay, launches that overlap)
// a 256^2 FP32 step takes 2.4 us, of which the collision is about 0.7 us; the rest is launch
// latency, the round trip of every population through L2 and the drain between launches.
// Here a step costs the collision, three block barriers and one exchange: 2.12 us at
// 256^2, 3.9 us at 512^2 (4.5 us by graph), FP64 64^2 7.7 us (15.9 us).  What is left
// at 256^2 (cycles): collision of the edge nodes 1500, sending them 600, the trip
// through L2 1200 to 1500, densities 400, barriers 200.  From about 400^2 on the
// collisions' issue bounds it.  Measured and not kept: 768 threads at 80 registers
// (2.77 against 2.45 us at 256^2); a fence and flags or a counter per step.
//
// The exchange carries its own arrival flag: three populations and the step's
// number form one 16-byte word (FP64: two words), written and read by single
// 128-bit accesses, so a reader that sees the number has the data.  No fence and
// no separate flag are needed; a fence plus a counter barrier measured 1.07 us per
// step on 152 blocks, more than the rest of the step.
//
// A tile needs of its surroundings what the pull and the density ring read: cells
// up to two nodes outside, and of those only the populations that move into the
// tile or its one-node ring.  Each tile publishes, for its left and right edges,
// the populations {0, 2, 4} and those leaving through that edge of the outermost
// column and the leaving ones of the next column, and the same for rows at its
// lower and upper edges (groups {0, 1, 3}); the corners of the ring come from the
// column groups of the diagonal tiles.  Words are double-buffered by the parity of
// the step: a tile writes step s + 2 only after reading every neighbour's step
// s + 1, which that neighbour sent after it had read step s.
//
// What the scratch buffer held before a run is never taken for a word of it: every tile
// clears its own words first, and no tile reads any before all tiles have (a grid barrier,
// arrived at right after clearing and waited for once the tile is loaded; waiting in the
// second step instead kept its state alive in the loop, 2.17 us a step at 256^2).  So handles
// that share a scratch buffer may run in turn, whatever they left in it.
#pragma once

#include <cooperative_groups.h>

#include <utility>

#include "lbm_tma.cuh"

namespace lbm {

constexpr int kResTiles = 152;              // at most one tile per SM
constexpr unsigned kResSmem = 227u * 1024;  // shared memory of a block
constexpr unsigned long long kResWaitNs = 10000000000ull;  // bound of an exchange wait (10 s)

template <typename T>
struct ResTraits;
template <>
struct ResTraits<float> {
  static constexpr int words = 1, max_threads = 512;
};
template <>
struct ResTraits<__half> {
  static constexpr int words = 1, max_threads = 512;
};
template <>
struct ResTraits<double> {
  static constexpr int words = 2, max_threads = 256;
};

// Node slots of a w x h tile, `lanes` nodes each: first the nodes within two of the
// tile's edge (those that are sent), then, from a whole warp on, the others.
struct ResSlots {
  int edge_nodes, edge;  // nodes and slots of the first kind
  int first;             // first slot of the second kind
  int inner_nodes, inner;
  int total;             // first + inner
};
__host__ __device__ __forceinline__ ResSlots res_slots(int w, int h, int lanes) {
  ResSlots s;
  s.inner_nodes = w > 4 && h > 4 ? (w - 4) * (h - 4) : 0;
  s.edge_nodes = w * h - s.inner_nodes;
  s.edge = (s.edge_nodes + lanes - 1) / lanes;
  s.inner = (s.inner_nodes + lanes - 1) / lanes;
  s.first = (s.edge + 31) / 32 * 32;
  s.total = s.first + s.inner;
  return s;
}
// Node k of slot q (k < lanes; a slot's missing last node repeats its first); false:
// an empty slot.
__host__ __device__ __forceinline__ bool res_node(const ResSlots& s, int w, int h, int q, int k, int& lx, int& ly) {
  if (q >= s.first) {
    int m = q - s.first + k * s.inner;
    if (m >= s.inner_nodes) m = q - s.first;
    const int r = m / (w - 4);
    ly = r + 2;
    lx = m - r * (w - 4) + 2;
    return true;
  }
  if (q >= s.edge) return false;
  int m = q + k * s.edge;
  if (m >= s.edge_nodes) m = q;
  if (s.inner_nodes == 0 || m < 2 * w) {  // all rows of a tile that is all edge, or the lower two
    ly = m / w;
    lx = m - ly * w;
  } else if (m < 4 * w) {  // the upper two rows
    m -= 2 * w;
    ly = m / w;
    lx = m - ly * w;
    ly += h - 2;
  } else {  // two columns at each side
    m -= 4 * w;
    const int side = m >= 2 * (h - 4);
    if (side) m -= 2 * (h - 4);
    ly = 2 + (m >> 1);
    lx = (m & 1) + (side ? w - 2 : 0);
  }
  return true;
}

// Bytes of the exchange tables (6 (h + w) + 6 (h + 4) + 6 w entries of 8 bytes) and
// the slot table (4 bytes a slot, at most one per `lanes` nodes and 33 more), a
// multiple of 16.
__host__ __device__ __forceinline__ int res_table_bytes(int wmax, int hmax, int lanes) {
  return ((12 * (wmax + hmax) + 24) * 8 + (wmax * hmax / lanes + 34) * 4 + 15) / 16 * 16;
}

// Arguments of the launch.
template <typename S>
struct ResArgs {
  const S* fin;        // state the run starts from
  S* fout;             // state after the last step (may be fin: see k_resident)
  S* rec;              // or null: the states after `rec_first` steps and every rec_every after
  long long rec_stride;  // go here, rec_stride elements apart
  int rec_first, rec_every;
  uint4* mail;         // exchange words, two parities
  int* err;
  unsigned step0;      // time step number of step 0 (seeds the FP16 rounding)
  int nsteps, nx, ny, gx, gy, wmax, hmax, pitch;
  int stochastic;
  Strides st;
};

// 16-byte words: one 128-bit access each way, so that the four parts arrive together.
__device__ __forceinline__ void st_word(uint4* p, uint4 v) {
  asm volatile(
      "{\n .reg .b64 a, b;\n .reg .b128 q;\n mov.b64 a, {%1, %2};\n mov.b64 b, {%3, %4};\n mov.b128 q, {a, b};\n"
      " st.relaxed.gpu.global.b128 [%0], q;\n}\n" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
      : "memory");
}
__device__ __forceinline__ uint4 ld_word(const uint4* p) {
  uint4 v;
  asm volatile(
      "{\n .reg .b64 a, b;\n .reg .b128 q;\n ld.relaxed.gpu.global.b128 q, [%4];\n mov.b128 {a, b}, q;\n"
      " mov.b64 {%0, %1}, a;\n mov.b64 {%2, %3}, b;\n}\n"
      : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
      : "l"(p)
      : "memory");
  return v;
}

// Population triples of the groups, four bits each: columns {0, 2, 4}, leaving left
// {3, 6, 7}, leaving right {1, 5, 8}; rows {0, 1, 3}, leaving down {4, 7, 8}, up {2, 5, 6}.
constexpr unsigned kTripX0 = 0x420, kTripXm = 0x763, kTripXp = 0x851;
constexpr unsigned kTripY0 = 0x310, kTripYm = 0x874, kTripYp = 0x652;

// Word index of a published group within its tile's block of 6 (hmax + wmax) groups.
// Columns: side 0 = left edge, 1 = right edge; k = 0, 1: the outermost column's two
// groups, 2: the next column's leaving group; y = local row.  Rows alike.
__host__ __device__ __forceinline__ int res_col_group(int side, int k, int y, int hmax) {
  return (side * 3 + k) * hmax + y;
}
__host__ __device__ __forceinline__ int res_row_group(int side, int k, int x, int hmax, int wmax) {
  return 6 * hmax + (side * 3 + k) * wmax + x;
}

__host__ __device__ __forceinline__ int res_lo(int b, int n, int g) { return int((long long)b * n / g); }

// One entry of the exchange tables: word index, cell offset and triple.
struct ResItem {
  unsigned word;
  unsigned cell;  // offset | triple << 16
};

// Entry r of a w x h tile's send list (6 (h + w) entries) and receive list
// (6 (h + 4) + 6 w entries).  pitch: row pitch of the shared arrays, whose cell
// (x, y) sits at (y + 2) pitch + x + 2.
__host__ __device__ __forceinline__ ResItem res_send_item(int r, int tile, int w, int h, int hmax, int wmax, int pitch) {
  const int groups = 6 * (hmax + wmax);
  ResItem it;
  int x, y;
  unsigned trip;
  if (r < 6 * h) {
    const int q = r / h, side = q / 3, k = q - 3 * side;
    y = r - q * h;
    x = side ? w - 1 - (k == 2) : (k == 2);
    trip = k == 0 ? kTripX0 : (side ? kTripXp : kTripXm);
    it.word = unsigned(tile * groups + res_col_group(side, k, y, hmax));
  } else {
    r -= 6 * h;
    const int q = r / w, side = q / 3, k = q - 3 * side;
    x = r - q * w;
    y = side ? h - 1 - (k == 2) : (k == 2);
    trip = k == 0 ? kTripY0 : (side ? kTripYp : kTripYm);
    it.word = unsigned(tile * groups + res_row_group(side, k, x, hmax, wmax));
  }
  it.cell = unsigned((y + 2) * pitch + x + 2) | trip << 16;
  return it;
}

__host__ __device__ __forceinline__ ResItem res_recv_item(int r, int bx, int by, int gx, int gy, int nx, int ny,
                                                          int hmax, int wmax, int pitch) {
  const int groups = 6 * (hmax + wmax);
  const int w = res_lo(bx + 1, nx, gx) - res_lo(bx, nx, gx), h = res_lo(by + 1, ny, gy) - res_lo(by, ny, gy);
  ResItem it;
  int x, y;
  unsigned trip;
  if (r < 6 * (h + 4)) {
    const int q = r / (h + 4), side = q / 3, k = q - 3 * side;  // side 0: halo columns right of the tile
    y = r - q * (h + 4) - 2;
    x = side ? (k == 2 ? -2 : -1) : (k == 2 ? w + 1 : w);
    trip = k == 0 ? kTripX0 : (side ? kTripXp : kTripXm);
    const int tx = side ? (bx == 0 ? gx - 1 : bx - 1) : (bx == gx - 1 ? 0 : bx + 1);
    int ty = by, ly = y;
    if (y < 0) {
      ty = by == 0 ? gy - 1 : by - 1;
      ly = y + res_lo(ty + 1, ny, gy) - res_lo(ty, ny, gy);
    } else if (y >= h) {
      ty = by == gy - 1 ? 0 : by + 1;
      ly = y - h;
    }
    it.word = unsigned((ty * gx + tx) * groups + res_col_group(side, k, ly, hmax));
  } else {
    r -= 6 * (h + 4);
    const int q = r / w, side = q / 3, k = q - 3 * side;  // side 0: halo rows above the tile
    x = r - q * w;
    y = side ? (k == 2 ? -2 : -1) : (k == 2 ? h + 1 : h);
    trip = k == 0 ? kTripY0 : (side ? kTripYp : kTripYm);
    const int ty = side ? (by == 0 ? gy - 1 : by - 1) : (by == gy - 1 ? 0 : by + 1);
    it.word = unsigned((ty * gx + bx) * groups + res_row_group(side, k, x, hmax, wmax));
  }
  it.cell = unsigned((y + 2) * pitch + x + 2) | trip << 16;
  return it;
}

// Words of a group.
__device__ __forceinline__ void res_send(uint4* mail, unsigned word, const float* p, int plane, unsigned trip,
                                         unsigned number) {
  st_word(mail + word, make_uint4(__float_as_uint(p[(trip & 15u) * plane]), __float_as_uint(p[(trip >> 4 & 15u) * plane]),
                                  __float_as_uint(p[(trip >> 8) * plane]), number));
}
__device__ __forceinline__ void res_send(uint4* mail, unsigned word, const __half* p, int plane, unsigned trip,
                                         unsigned number) {
  st_word(mail + word, make_uint4(__half_as_ushort(p[(trip & 15u) * plane]), __half_as_ushort(p[(trip >> 4 & 15u) * plane]),
                                  __half_as_ushort(p[(trip >> 8) * plane]), number));
}
__device__ __forceinline__ void res_send(uint4* mail, unsigned word, const double* p, int plane, unsigned trip,
                                         unsigned number) {
  const double a = p[(trip & 15u) * plane], b = p[(trip >> 4 & 15u) * plane], c = p[(trip >> 8) * plane];
  st_word(mail + 2 * word, make_uint4(__double2loint(a), __double2hiint(a), __double2loint(b), number));
  st_word(mail + 2 * word + 1, make_uint4(__double2loint(c), __double2hiint(c), __double2hiint(b), number));
}
// A group's words as read, and their cells when every word holds `number` (else false).
template <int W>
struct ResWords {
  uint4 v[W];
};
template <int W>
__device__ __forceinline__ ResWords<W> res_load(const uint4* mail, unsigned word) {
  ResWords<W> r;
#pragma unroll
  for (int k = 0; k < W; ++k) r.v[k] = ld_word(mail + size_t(W) * word + k);
  return r;
}
__device__ __forceinline__ bool res_put(const ResWords<1>& r, float* p, int plane, unsigned trip, unsigned number) {
  if (r.v[0].w != number) return false;
  p[(trip & 15u) * plane] = __uint_as_float(r.v[0].x);
  p[(trip >> 4 & 15u) * plane] = __uint_as_float(r.v[0].y);
  p[(trip >> 8) * plane] = __uint_as_float(r.v[0].z);
  return true;
}
__device__ __forceinline__ bool res_put(const ResWords<1>& r, __half* p, int plane, unsigned trip, unsigned number) {
  if (r.v[0].w != number) return false;
  p[(trip & 15u) * plane] = __ushort_as_half((unsigned short)r.v[0].x);
  p[(trip >> 4 & 15u) * plane] = __ushort_as_half((unsigned short)r.v[0].y);
  p[(trip >> 8) * plane] = __ushort_as_half((unsigned short)r.v[0].z);
  return true;
}
__device__ __forceinline__ bool res_put(const ResWords<2>& r, double* p, int plane, unsigned trip, unsigned number) {
  const uint4 v = r.v[0], u = r.v[1];
  if (v.w != number || u.w != number) return false;
  p[(trip & 15u) * plane] = __hiloint2double(v.y, v.x);
  p[(trip >> 4 & 15u) * plane] = __hiloint2double(u.z, v.z);
  p[(trip >> 8) * plane] = __hiloint2double(u.y, u.x);
  return true;
}

__device__ __forceinline__ float res_get(const float* p) { return *p; }
__device__ __forceinline__ float res_get(const __half* p) { return __half2float(*p); }
__device__ __forceinline__ double res_get(const double* p) { return *p; }

// Storage value of population i of a node (FP16: the rounding of store9).
__device__ __forceinline__ float res_round(float v, unsigned, bool, int, float) { return v; }
__device__ __forceinline__ double res_round(double v, unsigned, bool, int, double) { return v; }
__device__ __forceinline__ __half res_round(float v, unsigned word, bool odd, int stochastic, __half) {
  if (!stochastic) return __float2half_rn(v);
  const unsigned h = cvt_rs_f16x2(odd ? 0.f : v, odd ? v : 0.f, word);
  return __ushort_as_half((unsigned short)(odd ? h >> 16 : h & 0xffffu));
}

// A value of V from one real per lane.
__device__ __forceinline__ f2 res_pack(const float (&a)[2]) { return f2{make_float2(a[0], a[1])}; }
__device__ __forceinline__ double res_pack(const double (&a)[1]) { return a[0]; }

// One step of the run, for a block and its tile (the phases of k_resident):
//   receive   the halo (first step: it came with the initial state)
//   phase 1b  densities of the edge nodes and the ring
//   phase 2   stencil and collision into the other buffer: the warps that own edge nodes
//             take those first, meet at a barrier of their own, send the edges, and then
//             take their share of the inner nodes
//   phase 1a  densities of the inner nodes, for the next step, with the first words of
//             the halo already asked for
// so that the words travel while the inner nodes are computed.
// Thread t owns slots t, t + T, ...  The arithmetic per node is that of the per-step
// kernels, so the result is the same bit for bit.
// fout == fin is allowed when nsteps >= 2: every tile that reads this tile's cells
// of fin has read them before it sends its first words, which this tile waits for
// before its second step.
template <typename V, typename S>
__global__ void __launch_bounds__(ResTraits<S>::max_threads, 1) k_resident(const ResArgs<S> a, const VCoef<V> c) {
  using real = typename LaneType<V>::type;
  constexpr int L = Lanes<V>::n;
  constexpr unsigned kEmpty = 0xffffffffu;
  extern __shared__ __align__(128) unsigned char dyn[];
  const int T = blockDim.x, tid = threadIdx.x;
  const int bx = blockIdx.x % a.gx, by = blockIdx.x / a.gx;
  const int x0 = res_lo(bx, a.nx, a.gx), y0 = res_lo(by, a.ny, a.gy);
  const int w = res_lo(bx + 1, a.nx, a.gx) - x0, h = res_lo(by + 1, a.ny, a.gy) - y0;
  const int pitch = a.pitch, plane = pitch * (a.hmax + 4);
  const int nsend = 6 * (h + w), nrecv = 6 * (h + 4) + 6 * w;
  const ResSlots sl = res_slots(w, h, L);
  // Shared memory: exchange tables, slot table, densities, two population buffers.
  ResItem* items = reinterpret_cast<ResItem*>(dyn);
  unsigned* slot = reinterpret_cast<unsigned*>(items + 12 * (a.wmax + a.hmax) + 24);
  real* rho = reinterpret_cast<real*>(dyn + res_table_bytes(a.wmax, a.hmax, L));
  S* cur = reinterpret_cast<S*>(rho + plane);
  S* nxt = cur + 9 * plane;
  constexpr int W = ResTraits<S>::words;
  const int own_words = 6 * (a.hmax + a.wmax) * W;  // of a tile, one parity
  const size_t mail_stride = size_t(a.gx) * a.gy * own_words;

  // This tile's words: number 0, which no step carries.  The barrier cannot block: the
  // launch is cooperative, and every block arrives before it waits for anything.
  for (int q = tid; q < 2 * own_words; q += T) {
    const bool odd = q >= own_words;
    st_word(a.mail + (odd ? mail_stride : 0) + size_t(blockIdx.x) * own_words + (q - (odd ? own_words : 0)),
            make_uint4(0u, 0u, 0u, 0u));
  }
  const cooperative_groups::grid_group grid = cooperative_groups::this_grid();
  auto cleared = grid.barrier_arrive();
  // Initial state of tile and halo (periodic), and the tables.
  for (int q = tid; q < (w + 4) * (h + 4); q += T) {
    const int ly = q / (w + 4), lx = q - ly * (w + 4);
    const int gx = wrap(x0 + lx - 2, a.nx), gy = wrap(y0 + ly - 2, a.ny);
    const S* p = a.fin + (gy * a.st.rs + gx);
#pragma unroll
    for (int i = 0; i < 9; ++i) cur[i * plane + ly * pitch + lx] = p[i * a.st.ps];
  }
  for (int r = tid; r < nsend; r += T) items[r] = res_send_item(r, blockIdx.x, w, h, a.hmax, a.wmax, pitch);
  for (int r = tid; r < nrecv; r += T)
    items[nsend + r] = res_recv_item(r, bx, by, a.gx, a.gy, a.nx, a.ny, a.hmax, a.wmax, pitch);
  for (int q = tid; q < sl.total; q += T) {  // cell offsets, lane 0 in the low half; read by this thread only
    unsigned v = 0;
    bool used = true;
#pragma unroll
    for (int k = 0; k < L; ++k) {
      int lx = 0, ly = 0;
      used = res_node(sl, w, h, q, k, lx, ly);
      v |= unsigned((ly + 2) * pitch + lx + 2) << (16 * k);
    }
    slot[q] = used ? v : kEmpty;
  }
  const int nring = 2 * (w + 2) + 2 * h;
  auto density_at = [&](const S* buf, int o) {
    real g[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) g[i] = res_get(buf + o + (i * plane - ey_of(i) * pitch - ex_of(i)));
    return sum9(g);
  };
  auto density = [&](const S* buf, int q) {  // of a slot
    const unsigned so = slot[q];
    if (so == kEmpty) return;
    if constexpr (L == 2) {
      const S* p0 = buf + (so & 0xffffu);
      const S* p1 = buf + (so >> 16);
      f2 d[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const int e = i * plane - ey_of(i) * pitch - ex_of(i);
        d[i].v = make_float2(res_get(p0 + e), res_get(p1 + e));
      }
      const f2 r = sum9(d);
      rho[so & 0xffffu] = r.v.x;
      rho[so >> 16] = r.v.y;
    } else {
      rho[so] = density_at(buf, int(so));
    }
  };
  const int inner_begin = tid >= sl.first ? tid : tid + (sl.first - tid + T - 1) / T * T;  // first inner slot of this thread
  const int senders = sl.first < T ? sl.first : T;  // threads that own edge slots (whole warps)
  // With one slot per thread, an inner warp lets the edge warp of its scheduler (warp
  // number modulo 4) go first: the edges then leave after the latency of one collision,
  // and the inner nodes follow while the words travel (256^2 FP32: 2.45 -> 2.15 us a step).
  const int edge_warps = senders / 32, warps = T / 32, warp = tid / 32;
  const int shared = edge_warps < 4 ? edge_warps : 4;  // schedulers with an edge warp
  const bool ordered = sl.total <= T && edge_warps < warps;
  const bool gated = ordered && warp >= edge_warps && (warp & 3) < shared;
  int gate_threads = 0;  // edge warps and the ones that wait for them
  for (int k = 0; k < warps; ++k) gate_threads += k < edge_warps || (k & 3) < shared ? 32 : 0;
  __syncthreads();
  for (int q = inner_begin; q < sl.total; q += T) density(cur, q);  // phase 1a of step 0
  grid.barrier_wait(std::move(cleared));

  S* rec = a.rec;
  int until = a.rec_first;  // steps until the next recorded state
  for (int s = 0;; ++s) {
    const unsigned number = unsigned(s);  // of the words read; step s sends s + 1
    bool late = false;
    if (s > 0) {
      // Two groups of this thread at a time; the first two are asked for before the
      // densities of the inner nodes, which hide the trip through L2.
      const uint4* mail = a.mail + (s & 1 ? mail_stride : 0);
      bool inner_done = false;
      for (int r0 = tid; r0 < nrecv || !inner_done; r0 += 2 * T) {
        const bool one = r0 < nrecv, two = r0 + T < nrecv;
        const ResItem i0 = items[nsend + (one ? r0 : 0)], i1 = items[nsend + (two ? r0 + T : 0)];
        ResWords<W> v0 = res_load<W>(mail, i0.word), v1 = res_load<W>(mail, i1.word);
        if (!inner_done) {
          for (int q = inner_begin; q < sl.total; q += T) density(cur, q);  // phase 1a
          inner_done = true;
        }
        bool d0 = !one, d1 = !two;
        unsigned long long t0 = 0;
        for (int polls = 0;; ++polls) {
          if (!d0) d0 = res_put(v0, cur + (i0.cell & 0xffffu), plane, i0.cell >> 16, number);
          if (!d1) d1 = res_put(v1, cur + (i1.cell & 0xffffu), plane, i1.cell >> 16, number);
          if (d0 && d1) break;
          if ((polls & 255) == 255) {
            const unsigned long long now = global_ns();
            if (t0 == 0) t0 = now;
            if (now - t0 > kResWaitNs) {
              late = true;
              break;
            }
          }
          if (!d0) v0 = res_load<W>(mail, i0.word);
          if (!d1) v1 = res_load<W>(mail, i1.word);
        }
        if (late) break;
      }
    }
    if (__syncthreads_or(late)) {
      if (tid == 0) atomicExch(a.err, 1);
      return;
    }
    // Phase 1b; the ring from the last thread on (the first warps own the edge slots).
    for (int q = tid; q < sl.first; q += T) density(cur, q);
    for (int r = T - 1 - tid; r < nring; r += T) {
      int lx, ly;
      if (r < 2 * (w + 2)) {
        const bool top = r >= w + 2;
        lx = (top ? r - (w + 2) : r) - 1;
        ly = top ? h : -1;
      } else {
        const int q = r - 2 * (w + 2);
        const bool right = q >= h;
        ly = right ? q - h : q;
        lx = right ? w : -1;
      }
      const int o = (ly + 2) * pitch + lx + 2;
      rho[o] = density_at(cur, o);
    }
    __syncthreads();
    // Phase 2.
    const bool last = s + 1 == a.nsteps;
    const bool record = rec != nullptr && --until == 0;
    const unsigned seed = sizeof(S) == 2 ? step_seed(a.step0 + unsigned(s)) : 0u;
    if (gated) asm volatile("bar.sync 2, %0;" ::"r"(gate_threads) : "memory");
    for (int q = tid; q < sl.total; q += T) {
      const unsigned so = slot[q];
      if (so != kEmpty) {
        int o[L];
#pragma unroll
        for (int k = 0; k < L; ++k) o[k] = int(so >> (16 * k) & 0xffffu);
        auto at = [&](int dy, int dx) {
          real v[L];
#pragma unroll
          for (int k = 0; k < L; ++k) v[k] = rho[o[k] + dy * pitch + dx];
          return res_pack(v);
        };
        const V ml = at(-1, -1), mc = at(-1, 0), mr = at(-1, 1), cl = at(0, -1), cr = at(0, 1);
        const V pl = at(1, -1), pc = at(1, 0), pr = at(1, 1);
        V d[9], out[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          real v[L];
#pragma unroll
          for (int k = 0; k < L; ++k) v[k] = res_get(cur + o[k] + (i * plane - ey_of(i) * pitch - ex_of(i)));
          d[i] = res_pack(v);
        }
        collide_node(c, lattice_part(c), d, at(0, 0), ml, mc, mr, cl, cr, pl, pc, pr, out);
#pragma unroll
        for (int k = 0; k < L; ++k) {
          int gx = 0, gy = 0;
          if (last || record || sizeof(S) == 2) {
            gy = o[k] / pitch;
            gx = x0 + (o[k] - gy * pitch) - 2;
            gy += y0 - 2;
          }
          unsigned rs = sizeof(S) == 2 ? sr_start(gx, gy, a.nx, seed) : 0u;
          S v[9];
#pragma unroll
          for (int i = 0; i < 9; ++i) {
            v[i] = res_round(Lanes<V>::get(out[i], k), sizeof(S) == 2 ? sr_next(rs) : 0u, gx & 1, a.stochastic, S(0));
            nxt[o[k] + i * plane] = v[i];
          }
          const int g = gy * a.st.rs + gx;
          if (last) {
#pragma unroll
            for (int i = 0; i < 9; ++i) a.fout[g + i * a.st.ps] = v[i];
          }
          if (record) {
#pragma unroll
            for (int i = 0; i < 9; ++i) rec[g + i * a.st.ps] = v[i];
          }
        }
      }
      if (ordered && q < sl.first) asm volatile("bar.arrive 2, %0;" ::"r"(gate_threads) : "memory");
      if (!last && q < sl.first && q + T >= sl.first) {
        // This thread's last edge slot: the edge warps meet and send.
        asm volatile("bar.sync 1, %0;" ::"r"(senders) : "memory");
        uint4* mail = a.mail + (s & 1 ? 0 : mail_stride);
        for (int r = tid; r < nsend; r += senders) {
          const ResItem it = items[r];
          res_send(mail, it.word, nxt + (it.cell & 0xffffu), plane, it.cell >> 16, number + 1u);
        }
      }
    }
    if (last) break;
    if (record) {
      rec += a.rec_stride;
      until = a.rec_every;
    }
    __syncthreads();
    S* t = cur;
    cur = nxt;
    nxt = t;
  }
}

}  // namespace lbm
