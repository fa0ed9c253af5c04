// C ABI of the coupled IBM-LBM step (include/ibm_lbm.h): handle lifetime,
// device memory, host<->device conversion, validation, and the step loop
// (CUDA graphs of 64 and 16 steps of collision and coupling, or of 16 steps
// and single steps of the separate kernels; see Path below).
#include <cuda_runtime.h>

#include <sys/mman.h>
#include <unistd.h>

#include <algorithm>
#include <array>
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <thread>
#include <unordered_map>
#include <vector>

#include "../../include/ibm_lbm.h"
#include "cluster_body.cuh"
#include "common.cuh"
#include "handle.h"
#include "internal.h"
#include "transfer_group.cuh"

using namespace ibm;

static_assert(BODY_GROUP <= XFER_GROUP_MAX && TRACER_GROUP <= XFER_GROUP_MAX,
              "transfer groups must fit the shared-memory marker records");

namespace {

int fail(ibm_lbm_t* h, int code, const std::string& msg) {
  if (h) h->err = msg;
  return code;
}

// No C++ exception crosses the C ABI: every entry point runs its body under
// this guard; a failed host allocation returns E_NOMEM, any other exception
// (e.g. a size the standard containers reject) E_ARG.
template <class F>
int abi_guard(ibm_lbm_t* h, F&& body) noexcept {
  const char* msg = nullptr;
  int code = IBM_LBM_OK;
  try {
    return body();
  } catch (const std::bad_alloc&) {
    code = IBM_LBM_E_NOMEM;
    msg = "host allocation failed";
  } catch (...) {
    code = IBM_LBM_E_ARG;
    msg = "invalid size or argument (host exception)";
  }
  if (h) {
    try {
      h->err = msg;
    } catch (...) {
    }
  }
  return code;
}

#define CUDA_TRY(h, call)                                                                   \
  do {                                                                                      \
    cudaError_t e_ = (call);                                                                \
    if (e_ != cudaSuccess)                                                                  \
      return fail((h), IBM_LBM_E_CUDA, std::string(#call ": ") + cudaGetErrorString(e_));   \
  } while (0)

void* dalloc(ibm_lbm_t* h, std::vector<Alloc>& pool, size_t bytes) {
  if (bytes == 0) bytes = 256;
  void* p = nullptr;
  if (h->has_alloc) {
    p = h->alloc.alloc(bytes, h->alloc.ctx);
  } else if (cudaMalloc(&p, bytes) != cudaSuccess) {
    cudaGetLastError();
    p = nullptr;
  }
  if (p) {
    pool.push_back({p, bytes});
    h->bytes += bytes;
  }
  return p;
}

// Whether every page of a host buffer is in memory (false if the system does
// not say).
bool pages_mapped(const void* p, size_t bytes, size_t page) {
  const size_t first = (size_t)p / page * page, last = (size_t)p + bytes;
  unsigned char in[256];
  for (size_t a = first; a < last; a += sizeof(in) * page) {
    const size_t n = std::min(sizeof(in), (last - a + page - 1) / page);
    if (mincore(reinterpret_cast<void*>(a), n * page, in) != 0) return false;
    for (size_t i = 0; i < n; ++i)
      if (!(in[i] & 1)) return false;
  }
  return true;
}

// Whether a caller's buffer is ordinary host memory. A copy also takes device,
// managed and pinned memory, whose pages are not to be touched from here.
bool pageable(const void* p) {
  cudaPointerAttributes a{};
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeUnregistered;
}

// Take the page faults of a host buffer before a copy, which would fault its
// pages one by one from the device's side: one byte per page is written (an
// output that is about to be overwritten) or read (an input), by several
// threads for a large buffer. A copy of 8 MB into fresh pages took 6 ms, and
// 0.25 ms into mapped ones; a page touched here costs ~0.25 us, or a cache
// miss if it was mapped. Below 64 KiB a copy is a few tens of us either way.
// Up to 16 MiB a buffer whose pages are all there is left alone: its copy takes
// less than the threads below (get_fields of a 77x94x67 lattice into arrays in
// use before: 0.14 of 1.88 ms of a two-step run).
void touch_pages(const void* p, size_t bytes, bool write) {
  if (!p || bytes < ((size_t)64 << 10)) return;
  const long pg = sysconf(_SC_PAGESIZE);
  const size_t page = pg > 0 ? (size_t)pg : 4096;
  if (bytes < ((size_t)16 << 20) && pages_mapped(p, bytes, page)) return;
  if (!pageable(p)) return;  // (asked last: ~2 us)
  // a thread for every 2 MiB (starting one costs as much as touching ~100 pages)
  const unsigned nt = std::min({8u, std::max(1u, std::thread::hardware_concurrency()), (unsigned)(bytes >> 21)});
  const size_t chunk = nt > 1 ? (bytes / nt + page - 1) / page * page : 0;
  auto touch = [p, page, write](size_t b, size_t e) {
    if (write) {
      volatile char* q = static_cast<volatile char*>(const_cast<void*>(p));
      for (size_t o = b; o < e; o += page) q[o] = 0;
    } else {
      const volatile char* q = static_cast<const volatile char*>(p);
      char sink = 0;
      for (size_t o = b; o < e; o += page) sink ^= q[o];
      (void)sink;
    }
  };
  std::vector<std::thread> th;
  size_t done = 0;  // [0, done) is handed to threads
  try {
    for (unsigned t = 0; t < nt && nt > 1; ++t) {
      const size_t b = t * chunk, e = std::min(bytes, b + chunk);
      if (b >= e) break;
      th.emplace_back(touch, b, e);
      done = e;
    }
  } catch (...) {
    // no more threads: the calling thread takes the rest (an optimisation only)
  }
  touch(done, bytes);
  for (auto& x : th) x.join();
}

void release_pool(ibm_lbm_t* h, std::vector<Alloc>& pool) {
  for (auto& a : pool) {
    if (h->has_alloc) h->alloc.release(a.p, h->alloc.ctx);
    else cudaFree(a.p);
    h->bytes -= a.bytes;
  }
  pool.clear();
}

void drop_graphs(ibm_lbm_t* h) {
  if (h->g_chunk) cudaGraphExecDestroy(h->g_chunk);
  h->g_chunk = nullptr;
  for (auto& row : h->g_single)
    for (auto& g : row) {
      if (g) cudaGraphExecDestroy(g);
      g = nullptr;
    }
  for (auto& g : h->g_mid) {
    if (g) cudaGraphExecDestroy(g);
    g = nullptr;
  }
}

int tiles(const LatticeDev& L) { return L.ntx * L.nty * L.ntz; }

// How the markers and the lattice exchange velocities and forces. SEPARATE:
// forces, spreading and interpolation as kernels of their own. FUSED (many
// membranes) and CLUSTER (few bodies, rigid or membranes): one kernel between
// two collisions does the interpolation and advection of a step and the forces
// and spreading of the next, into the force density (and, for CLUSTER, the
// tile flags) that the next collision reads; the buffers alternate.
enum Path { SEPARATE, FUSED, CLUSTERED };

// Up to how many membranes of nv vertices clusters pay. One block per body
// (couple.cu; over ~938 vertices the separate kernels) does less work in all,
// but its latency decides while the bodies do not fill the chip, the more so
// the larger the template. us a step in a lattice with n bodies, clusters / one
// block (152 SMs: 15 clusters at one block an SM, 36 at two):
//   vertices     n = 1       n = 15      n = 16      n = 36      n = 38
//     42      30.1/29.0   35.8/32.4   37.0/31.6   43.5/35.3   65.9/35.2
//    162      33.1/32.2   38.3/35.3   40.2/34.8   46.9/38.4   71.3/38.3
//    362      34.4/37.5   39.6/40.9   42.3/40.6   48.4/44.4   77.0/44.2
//    642      36.3/43.8   41.2/47.7   44.8/47.5   51.6/51.8   81.6/51.9
//   1442      42.0/71.7   47.4/79.5   52.5/79.8   59.6/83.7   94.4/83.7
//   2562      49.7/91.7   53.8/96.9   82.9/96.9    101/101     126/101
// Beside rigid bodies, and in a server, there is no kernel of one block per
// body that couples, only the separate ones: clusters are better in one wave.
// A server's wave is that of all its cases. A case's path must not depend on
// what else is served, so the slots count, not the cases there are. us a step,
// clusters / separate, cases x membranes of 642 vertices: 8 x 1 55.5/76.8, 8 x 3
// 62.2/79.7, 32 x 1 153/169, 16 x 3 138/117, 8 x 8 108/86.1, 64 x 1 299/275, 64 x 8
// 804/393 (a server of 64 slots may hold few: 4 x 1 44.5/62.8).
constexpr int SERVED_MAX = 64;
int membrane_clusters_max(const ibm_lbm_t* h, int nv) {
  if (h->served_slots > 0) return (nv >= 512 && h->n_membranes == 1 ? SERVED_MAX : h->clusters_two) / h->served_slots;
  if (nv >= 512 || h->n_rigids > 0) return h->clusters_two;
  return nv >= 256 ? h->clusters_one : 0;
}
// Up to how many rigid bodies of [least, most] markers clusters pay against the
// separate kernels (a block per body and stage). us a step in a lattice with n
// tethered bodies, clusters / separate:
//   markers      n = 1      n = 28      n = 38      n = 57      n = 72      n = 76     n = 1000
//     92      15.7/34.4  20.3/35.1   34.9/35.1   35.8/35.5   49.9/35.7   51.0/35.9   471/153
//    362      20.2/47.3  28.3/52.0   47.8/51.9   49.2/52.1   58.6/55.6   71.1/55.8   700/305
//    812      21.1/63.5  30.3/70.6   53.0/70.6   53.8/71.5   63.1/75.4   78.4/75.4   784/395
//   2562      36.8/92.0  53.3/101    97.0/101    98.5/122     108/139     137/139
//   4002      49.4/111   72.3/119     132/120     135/155     147/164     187/164
// and direct forcing, whose clusters wait for the new pose before they spread:
//    362      30.3/49.2  39.9/54.6   70.3/54.8   72.9/55.3   81.8/58.8    101/58.6   998/326
//    812      32.2/70.3  42.8/75.5   76.0/75.6   78.9/76.2   86.6/80.1    109/80.0  1064/422
// One wave of clusters always wins; two (half a second one from 256 markers)
// win for tethered bodies of a size that is neither launch-bound nor a large
// scatter, but not beside membranes, whose clusters run after them while the
// separate kernels take both at once (5 membranes of 642 vertices and 20 bodies
// of 812: 77.9/91.6 us a step, and 40: 99.1/91.5). In a server of shear cells with one body each (24^3 to 64^3), cells of
// 92 and of 812 markers: 24 118/130 and 121/163, 48 215/207 and 223/241, 64 277/257
// and 283/292, 80 349/323 and 365/359, 128 538/485 and 557/521, 512 1962/1749 and
// 2031/1866; eight bodies of 812 markers in 8 cells 78.1/90.3, in 16 161/125: up to
// 64 bodies over its slots.
int rigid_clusters_max(const ibm_lbm_t* h, int least, int most, bool direct) {
  if (h->served_slots > 0) return SERVED_MAX / h->served_slots;
  const int two = h->clusters_two;
  if (direct || least < 256 || most > 3072 || h->n_membranes > 0) return two;
  return least < 512 ? two + two / 2 : 2 * two;
}
// Steps of the solid-only dynamics in one launch of clusters, and up to how
// many membranes of nv vertices they take it. A wave holds clusters_one of them
// (a block on an SM each), and takes 7 us a step (42 vertices) to 14 (2562); the
// general path (a block per body, three launches) grows slowly with the count.
// us a step, clusters / general:
//   vertices    n = 15     n = 30     n = 45     n = 60     n = 75     n = 90     n = 120
//     42       6.9/15.6  13.7/16.8  20.5/16.7  27.2/16.6  34.0/17.0  40.8/17.4  54.3/16.6
//    252       7.2/19.7  14.3/20.7  21.2/20.4  28.4/22.8  35.4/22.8  42.3/22.8  56.4/26.9
//    642       8.4/26.9  16.5/28.9  24.6/33.0  32.8/33.0  40.9/35.1  49.0/39.2  65.2/41.5
//   1442      11.4/41.0  22.6/47.2  34.0/53.3  45.1/55.6  56.3/61.9  67.7/66.7  89.9/77.3
//   2562      14.4/60.1  28.6/70.4  42.8/80.3  57.0/85.9  71.2/95.6   85.3/105   113/122
constexpr int64_t SOLID_CHUNK = 512;
int solid_clusters_max(const ibm_lbm_t* h, int nv) { return (2 + nv / 400) * h->clusters_one; }

Path path_of(const ibm_lbm_t* h) {
  if (h->m.M == 0 || h->morse_rc > 0.0) return SEPARATE;
  if (h->cluster_boxes) return CLUSTERED;
  return h->n_couple > 0 ? FUSED : SEPARATE;
}

// Lattice view of a step that uses force-density buffer k (0 or 1).
LatticeDev lattice_of(const ibm_lbm_t* h, Path p, int k) {
  LatticeDev L = h->L;
  if (p != SEPARATE && k) L.g = h->gbuf2;
  if (p == CLUSTERED && k) L.flags = h->fbuf2;
  return L;
}

// Whether a collision and the coupling by clusters start ahead of one another
// (await_predecessor): one kernel each (rigid bodies or membranes alone, a
// lattice with fluid), nothing timed between them, and a small lattice: at 32^3
// a step goes from 22.5 to 20.5 us, but blocks that wait in residence cost a
// collision of many waves more than the gap between two kernels (256^3 tube:
// 187 -> 206 ms per 200 steps). Nor where the clusters fill the device: blocks
// of a collision that waits take the places of some, which then run as a second
// wave (60^3, 36 tethered bodies of 812 markers: 52 us a step, ordered 33).
bool chained(const ibm_lbm_t* h) {
  return !h->timing && h->n_rows > 0 && h->L.N <= CHAINED_CELLS_MAX && (h->n_rigids > 0) != (h->n_membranes > 0) &&
         leaves_room(h->n_rigids + h->n_membranes, h->clusters_two);
}

// Blocks of n clusters on an SM: one while they are all resident so, for
// larger boxes.
int per_sm(const ibm_lbm_t* h, int n) { return n <= h->clusters_one ? 1 : CLUSTER_PER_SM; }

void enqueue_cluster(ibm_lbm_t* h, int k, int next, bool interp, bool forces, bool spread) {
  const LatticeDev L = lattice_of(h, CLUSTERED, k), Ln = lattice_of(h, CLUSTERED, next);
  launch_couple_cluster(L, Ln.g, Ln.flags, h->m, h->d_bodies, h->rigid_list, h->n_rigids, false, h->cluster_max,
                        h->mesh, h->cluster_boxes, per_sm(h, h->n_rigids), interp, forces, spread,
                        interp && chained(h), h->stream);
  launch_couple_cluster(L, Ln.g, Ln.flags, h->m, h->d_bodies, h->membrane_list, h->n_membranes, true, h->mesh.nv,
                        h->mesh, h->cluster_boxes, per_sm(h, h->n_membranes), interp, forces, spread,
                        interp && chained(h), h->stream);
}

// Marker forces: each body's own forces (membranes, rigid tethers,
// filaments), then the Morse excluded volume between bodies.
void enqueue_forces(ibm_lbm_t* h, cudaStream_t st) {
  if (h->m.M == 0) return;
  if (h->cluster_boxes)
    enqueue_cluster(h, 0, 0, false, true, false);
  else
    launch_forces(h->m, h->d_bodies, h->membrane_list, h->n_membranes, h->rigid_list, h->n_rigids, h->mesh, st);
  launch_filaments(h->m, h->d_bodies, h->filament_list, h->n_filaments, st);
  if (h->morse_rc > 0.0 && h->morse_ready)
    launch_morse(h->morse, h->m, h->cfg.nx, h->cfg.ny, h->cfg.nz, h->cfg.geometry, st);
}

// Spreading of the bodies' forces and the tiles of the tracers' stencils (whose
// forces a step has zeroed).
void spread(ibm_lbm_t* h, const LatticeDev& L) {
  launch_spread(L, h->m, h->groups, h->n_body_groups, h->boxes, h->stream);
  if (!h->tracers_everywhere)
    launch_tracers_mark(L, h->m, h->groups + h->n_body_groups, h->n_groups - h->n_body_groups, h->stream);
}

void interpolate(ibm_lbm_t* h, const LatticeDev& L) {
  launch_interpolate(L, h->m, h->groups, h->n_body_groups, h->boxes, h->stream);
  launch_tracers_move(L, h->m, h->groups + h->n_body_groups, h->n_groups - h->n_body_groups, h->stream);
}

// Forces and spreading of the first step into buffer k.
void couple_begin(ibm_lbm_t* h, Path p, int k) {
  cudaStream_t st = h->stream;
  const LatticeDev L = lattice_of(h, p, k);
  cudaMemsetAsync(h->fbuf, 0, (size_t)tiles(L), st);
  if (h->m.M == 0) return;
  if (p == CLUSTERED) {
    cudaMemsetAsync(h->fbuf2, 0, (size_t)tiles(L), st);
    enqueue_cluster(h, k, k, false, true, true);
    return;
  }
  enqueue_forces(h, st);
  spread(h, L);
}

// Interpolation and advection of the step that used buffer k, forces and
// spreading of the next into the other one.
void couple_mid(ibm_lbm_t* h, Path p, int k) {
  if (p == CLUSTERED) {
    enqueue_cluster(h, k, k ^ 1, true, true, true);
    return;
  }
  const LatticeDev L = lattice_of(h, p, k);
  cudaMemsetAsync(L.flags, 0, (size_t)tiles(L), h->stream);
  launch_couple(L, k ? h->gbuf : h->gbuf2, h->m, h->d_bodies, h->couple_items, h->n_couple, h->groups, h->boxes,
                h->couple_order, h->mesh, h->stream);
}

// Interpolation and advection of the last step.
void couple_end(ibm_lbm_t* h, Path p, int k) {
  if (h->m.M == 0) return;
  if (p == CLUSTERED) enqueue_cluster(h, k, k, true, false, false);
  else interpolate(h, lattice_of(h, p, k));
}

void collide(ibm_lbm_t* h, Path p, int k, bool odd, bool dense) {
  const bool early = p == CLUSTERED && chained(h);  // a coupling comes right before
  launch_collide(lattice_of(h, p, k), h->rows, h->n_rows, h->cfg.storage, odd, dense || h->tracers_everywhere, early,
                 h->stream);
}

// One coupled step by itself on the handle's stream (also used under
// capture); it needs the first buffers only. With `waiting`, a force density
// that a SPREAD stage left in the first buffer goes into this step wherever it
// lies (every tile is read) and is gone after it: the couplings clear what
// they spread themselves.
void enqueue_step(ibm_lbm_t* h, bool odd, bool dense, bool waiting = false) {
  const Path p = path_of(h);
  couple_begin(h, p, 0);
  if (waiting) cudaMemsetAsync(h->fbuf, 1, (size_t)tiles(h->L), h->stream);
  collide(h, p, 0, odd, dense);
  if (waiting) cudaMemsetAsync(h->gbuf, 0, sizeof(float4) * (size_t)h->L.N, h->stream);
  couple_end(h, p, 0);
}

// One step with an event before each stage and after the last.
void enqueue_timed_step(ibm_lbm_t* h, bool odd, bool dense, bool waiting) {
  cudaStream_t st = h->stream;
  const size_t base = 5 * h->timed_steps;
  const bool rec = base + 5 <= h->events.size();
  auto mark = [&](int k) {
    if (rec) cudaEventRecord(h->events[base + k], st);
  };
  const LatticeDev L = h->L;
  mark(0);
  enqueue_forces(h, st);
  mark(1);
  cudaMemsetAsync(L.flags, 0, (size_t)tiles(L), st);
  if (h->m.M > 0) spread(h, L);
  if (waiting) cudaMemsetAsync(L.flags, 1, (size_t)tiles(L), st);
  mark(2);
  collide(h, SEPARATE, 0, odd, dense);
  mark(3);
  if (waiting) cudaMemsetAsync(L.g, 0, sizeof(float4) * (size_t)L.N, st);
  if (h->m.M > 0) interpolate(h, L);
  mark(4);
  if (rec) {
    h->timed_odd.push_back(odd ? 1 : 0);
    h->timed_fused.push_back(0);
    h->timed_steps++;
  }
}

int end_capture(ibm_lbm_t* h, cudaGraphExec_t* out) {
  cudaGraph_t g = nullptr;
  CUDA_TRY(h, cudaStreamEndCapture(h->stream, &g));
  cudaError_t e = cudaGraphInstantiate(out, g, 0);
  cudaGraphDestroy(g);
  if (e != cudaSuccess) return fail(h, IBM_LBM_E_CUDA, std::string("cudaGraphInstantiate: ") + cudaGetErrorString(e));
  return IBM_LBM_OK;
}

int capture(ibm_lbm_t* h, cudaGraphExec_t* out, int n, bool odd0, bool dense_last) {
  CUDA_TRY(h, cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal));
  bool odd = odd0;
  for (int s = 0; s < n; ++s) {
    enqueue_step(h, odd, dense_last && s == n - 1);
    odd = !odd;
  }
  return end_capture(h, out);
}

// n times (even) collision and coupling into the next step, from an even
// step on: step parity and buffer alternate together.
int capture_mid(ibm_lbm_t* h, Path p, cudaGraphExec_t* out, int n) {
  CUDA_TRY(h, cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal));
  for (int s = 0; s < n; ++s) {
    collide(h, p, s & 1, (s & 1) != 0, false);
    couple_mid(h, p, s & 1);
  }
  return end_capture(h, out);
}

// Whether a call of n steps couples two steps with one kernel.
bool fused_applies(const ibm_lbm_t* h) {
  return path_of(h) != SEPARATE && (!h->timing || h->timing_fused) && h->gbuf2 != nullptr;
}

// n coupled steps on a fused path, the last one with the moments of every
// cell if dense: the first step's forces and spreading, then collision and
// coupling by turns, the last step's interpolation alone. With timed, the
// steps that launch the coupling kernel record events around the collision
// and around the coupling (the forces and spreading slots of such a step are
// not read); kernels are then launched directly.
int enqueue_fused(ibm_lbm_t* h, int64_t n, bool dense, bool timed) {
  cudaStream_t st = h->stream;
  const Path p = path_of(h);
  int k = h->odd_next ? 1 : 0;  // the buffer goes with the AA parity
  couple_begin(h, p, k);
  int64_t mids = n - 1;
  while (mids > 0) {
    const int which = mids >= FUSED_LONG ? 0 : 1, len = which == 0 ? FUSED_LONG : CHUNK;
    if (!timed && k == 0 && mids >= len) {
      if (!h->g_mid[which]) {
        const int rc = capture_mid(h, p, &h->g_mid[which], len);
        if (rc) return rc;
      }
      CUDA_TRY(h, cudaGraphLaunch(h->g_mid[which], st));
      mids -= len;
        continue;
    }
    const size_t base = 5 * h->timed_steps;
    const bool rec = timed && base + 5 <= h->events.size();
    if (rec) cudaEventRecord(h->events[base + 2], st);
    collide(h, p, k, k != 0, false);
    if (rec) cudaEventRecord(h->events[base + 3], st);
    couple_mid(h, p, k);
    if (rec) {
      cudaEventRecord(h->events[base + 4], st);
      h->timed_odd.push_back(k != 0 ? 1 : 0);
      h->timed_fused.push_back(1);
      h->timed_steps++;
    }
    k ^= 1;
    --mids;
  }
  collide(h, p, k, k != 0, dense);
  couple_end(h, p, k);
  h->steps += n;
  if (n & 1) h->odd_next = !h->odd_next;
  return IBM_LBM_OK;
}

int enqueue_diagnostics(ibm_lbm_t* h) {
  cudaStream_t st = h->stream;
  CUDA_TRY(h, cudaMemsetAsync(h->d_diag, 0, 8 * sizeof(double), st));
  CUDA_TRY(h, cudaMemsetAsync(h->d_umax, 0, sizeof(unsigned), st));
  launch_diagnostics(h->L, h->rows, h->n_rows, h->d_diag, h->d_umax, st);
  CUDA_TRY(h, cudaGetLastError());
  CUDA_TRY(h, cudaMemcpyAsync(h->h_diag, h->d_diag, 8 * sizeof(double), cudaMemcpyDeviceToHost, st));
  CUDA_TRY(h, cudaMemcpyAsync(h->h_umax, h->d_umax, sizeof(unsigned), cudaMemcpyDeviceToHost, st));
  CUDA_TRY(h, cudaMemcpyAsync(h->h_status, h->L.status, sizeof(int), cudaMemcpyDeviceToHost, st));
  h->diag_pending = true;
  return IBM_LBM_OK;
}

int finish_diagnostics(ibm_lbm_t* h) {
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  if (!h->diag_pending) return IBM_LBM_OK;
  h->diag_pending = false;
  float umax2;
  std::memcpy(&umax2, h->h_umax, sizeof(float));
  if (*h->h_status != 0 || !std::isfinite(umax2) || umax2 > 0.16f) {
    char buf[160];
    std::snprintf(buf, sizeof buf, "unstable: non-finite moments or |u| > 0.4 (max |u|^2 = %g) after %lld steps",
                  (double)umax2, h->steps);
    return fail(h, IBM_LBM_E_UNSTABLE, buf);
  }
  return IBM_LBM_OK;
}

int enqueue_steps(ibm_lbm_t* h, int64_t n) {
  if (n < 0) return fail(h, IBM_LBM_E_ARG, "n_steps < 0");
  if (n == 0) return IBM_LBM_OK;
  h->boxes_valid = false;  // the last interpolation moves the markers
  // no force acts on the tracers (set_marker_forces may have left some)
  if (h->need_zero_F) CUDA_TRY(h, cudaMemsetAsync(h->m.F, 0, sizeof(float4) * (size_t)h->m.M, h->stream));
  int64_t left = n;
  if (path_of(h) != SEPARATE && !h->gbuf2 && (h->timing ? h->timing_fused && left > 2 : left > 1)) {
    if (!ensure_second_buffer(h)) CUDA_TRY(h, cudaGetLastError());  // (no memory: separate kernels)
  }
  const bool fused = fused_applies(h);
  if (h->density_waiting) {
    const bool odd = h->odd_next, dense = left == 1;
    if (h->timing && !fused) enqueue_timed_step(h, odd, dense, true);
    else enqueue_step(h, odd, dense, true);
    h->density_waiting = false;
    --left;
    h->steps += 1;
    h->odd_next = !odd;
  }
  if (h->timing) {
    // with timing_fused, a handle on a fused path times only its coupled
    // steps, the last one of the call apart; every other handle is timed
    // stage by stage
    while (left > 0) {
      if (fused && !h->odd_next && left > 2) {
        const int m = (int)std::min<int64_t>(left - 1, 1 << 22);
        const int rc = enqueue_fused(h, m, false, true);
        if (rc) return rc;
        left -= m;
        continue;
      }
      if (fused) enqueue_step(h, h->odd_next, left == 1);
      else enqueue_timed_step(h, h->odd_next, left == 1, false);
      --left;
      h->steps += 1;
      h->odd_next = !h->odd_next;
    }
    CUDA_TRY(h, cudaGetLastError());
    return enqueue_diagnostics(h);
  }
  if (fused && left > 1) {
    const int rc = enqueue_fused(h, left, true, false);
    if (rc) return rc;
    CUDA_TRY(h, cudaGetLastError());
    return enqueue_diagnostics(h);
  }
  while (left > 0) {
    if (!h->odd_next && left > CHUNK) {
      if (!h->g_chunk) {
        int rc = capture(h, &h->g_chunk, CHUNK, false, false);
        if (rc) return rc;
      }
      CUDA_TRY(h, cudaGraphLaunch(h->g_chunk, h->stream));
      left -= CHUNK;
      h->steps += CHUNK;
    } else {
      const int odd = h->odd_next ? 1 : 0, dense = (left == 1) ? 1 : 0;
      if (!h->g_single[odd][dense]) {
        int rc = capture(h, &h->g_single[odd][dense], 1, odd, dense);
        if (rc) return rc;
      }
      CUDA_TRY(h, cudaGraphLaunch(h->g_single[odd][dense], h->stream));
      left -= 1;
      h->steps += 1;
      h->odd_next = !h->odd_next;
    }
  }
  return enqueue_diagnostics(h);
}

// ---- membrane template: edges and rest state (FP64) --------------------------
struct HostMesh {
  std::vector<int4> edges;
  std::vector<int2> edge_tris;
  std::vector<float4> edge_rest;
  std::vector<int> v_edge_start, v_edge, v_tri_start, v_tri;
  std::vector<int4> tris;
  std::vector<float> area0;
  double A0 = 0, V0 = 0;
};

struct V3 {
  double x, y, z;
};
V3 sub(V3 a, V3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
V3 crs(V3 a, V3 b) { return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x}; }
double dt3(V3 a, V3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }

// Orders items (triangles or edges) so that, in each run of 32 consecutive
// items (one warp of the membrane force kernel), the vertices (and
// triangles) an item reads and accumulates into in each of its roles differ
// modulo 32: the warp's shared-memory accesses for one role then fall in
// distinct banks. Greedy: each run takes the first remaining items whose
// residues are all still free; a run that finds none completes with the
// items of fewest clashes. Only the order changes, not the items.
template <int R>
std::vector<int> bank_order(const std::vector<std::array<int, R>>& keys) {
  const int n = (int)keys.size();
  std::vector<int> order;
  order.reserve(n);
  std::vector<char> taken(n, 0);
  int left = n;
  while (left > 0) {
    uint32_t used[R] = {};
    int in_run = 0;
    for (int pass = 0; pass < 2 && in_run < 32 && in_run < left; ++pass) {
      for (int i = 0; i < n && in_run < 32 && in_run < left; ++i) {
        if (taken[i]) continue;
        int clash = 0;
        for (int r = 0; r < R; ++r) clash += (used[r] >> (keys[i][r] & 31)) & 1u;
        if (pass == 0 && clash) continue;
        taken[i] = 1;
        order.push_back(i);
        for (int r = 0; r < R; ++r) used[r] |= 1u << (keys[i][r] & 31);
        ++in_run;
      }
    }
    left -= in_run;
  }
  return order;
}

void order_for_banks(HostMesh& m) {
  // triangles: their three vertices
  std::vector<std::array<int, 3>> tk(m.tris.size());
  for (size_t t = 0; t < m.tris.size(); ++t) tk[t] = {m.tris[t].x, m.tris[t].y, m.tris[t].z};
  const std::vector<int> to = bank_order<3>(tk);
  std::vector<int> new_of_t(m.tris.size());
  std::vector<int4> tris(m.tris.size());
  for (size_t i = 0; i < to.size(); ++i) {
    tris[i] = m.tris[to[i]];
    new_of_t[to[i]] = (int)i;
  }
  m.tris.swap(tris);
  for (auto& et : m.edge_tris) et = make_int2(new_of_t[et.x], new_of_t[et.y]);
  // edges: their four vertices and two triangles
  std::vector<std::array<int, 6>> ek(m.edges.size());
  for (size_t e = 0; e < m.edges.size(); ++e)
    ek[e] = {m.edges[e].x, m.edges[e].y, m.edges[e].z, m.edges[e].w, m.edge_tris[e].x, m.edge_tris[e].y};
  const std::vector<int> eo = bank_order<6>(ek);
  std::vector<int4> edges(m.edges.size());
  std::vector<int2> et(m.edges.size());
  for (size_t i = 0; i < eo.size(); ++i) {
    edges[i] = m.edges[eo[i]];
    et[i] = m.edge_tris[eo[i]];
  }
  m.edges.swap(edges);
  m.edge_tris.swap(et);
}

// The part of a template that the vertices [v0, v1) need: every edge that has
// one of them among its four, with both its triangles (the forces on c and d
// need their normals), and every triangle that has one of them; those first.
struct MeshPartHost {
  std::vector<ushort4> edges, tris;
  std::vector<ushort2> edge_tris;
  std::vector<float4> edge_rest;
  std::vector<float> area0;
  int nt_own = 0;
};
MeshPartHost mesh_part_of(const HostMesh& m, int v0, int v1) {
  auto own = [&](int v) { return v >= v0 && v < v1; };
  MeshPartHost P;
  std::vector<int> touching, ghosts, edges;
  std::vector<int> local(m.tris.size(), -1);
  for (size_t t = 0; t < m.tris.size(); ++t)
    if (own(m.tris[t].x) || own(m.tris[t].y) || own(m.tris[t].z)) {
      touching.push_back((int)t);
      local[t] = 0;
    }
  for (size_t e = 0; e < m.edges.size(); ++e) {
    const int4 E = m.edges[e];
    if (!own(E.x) && !own(E.y) && !own(E.z) && !own(E.w)) continue;
    edges.push_back((int)e);
    for (int t : {m.edge_tris[e].x, m.edge_tris[e].y})
      if (local[t] < 0) {
        local[t] = 0;
        ghosts.push_back(t);
      }
  }
  // (in the template's order, which spreads the shared-memory banks)
  P.nt_own = (int)touching.size();
  std::vector<int> order = touching;
  order.insert(order.end(), ghosts.begin(), ghosts.end());
  for (size_t i = 0; i < order.size(); ++i) {
    const int t = order[i];
    local[t] = (int)i;
    P.tris.push_back(make_ushort4(m.tris[t].x, m.tris[t].y, m.tris[t].z, own(m.tris[t].x) ? 1 : 0));
    P.area0.push_back(m.area0[t]);
  }
  for (int e : edges) {
    const int4 E = m.edges[e];
    P.edges.push_back(make_ushort4(E.x, E.y, E.z, E.w));
    P.edge_tris.push_back(make_ushort2(local[m.edge_tris[e].x], local[m.edge_tris[e].y]));
    P.edge_rest.push_back(m.edge_rest[e]);
  }
  return P;
}

bool build_mesh(const ibm_lbm_mesh* mesh, HostMesh& out, std::string& why) {
  const int nv = mesh->n_vertices, nt = mesh->n_triangles;
  if (nv < 4 || nv > MAX_MESH_VERTICES || nt < 4 || !mesh->tris || !mesh->rest_X) {
    why = "mesh: need 4 <= n_vertices <= 4096, n_triangles >= 4 and both arrays";
    return false;
  }
  auto P = [&](int v) { return V3{mesh->rest_X[v], mesh->rest_X[nv + v], mesh->rest_X[2 * nv + v]}; };
  std::unordered_map<uint64_t, int> emap;
  out.edges.clear();
  out.edge_tris.clear();
  out.tris.resize(nt);
  for (int t = 0; t < nt; ++t) {
    int v[3] = {mesh->tris[3 * t], mesh->tris[3 * t + 1], mesh->tris[3 * t + 2]};
    for (int s = 0; s < 3; ++s)
      if (v[s] < 0 || v[s] >= nv) {
        why = "mesh: triangle vertex index out of range";
        return false;
      }
    out.tris[t] = make_int4(v[0], v[1], v[2], 0);
    for (int s = 0; s < 3; ++s) {
      const int a = v[s], b = v[(s + 1) % 3], c = v[(s + 2) % 3];
      const uint64_t key = ((uint64_t)std::min(a, b) << 32) | (uint32_t)std::max(a, b);
      auto it = emap.find(key);
      if (it == emap.end()) {
        emap.emplace(key, (int)out.edges.size());
        out.edges.push_back(make_int4(a, b, c, -1));
        out.edge_tris.push_back(make_int2(t, -1));
      } else {
        int4& e = out.edges[it->second];
        if (e.w >= 0 || e.x != b || e.y != a) {
          why = "mesh: not a closed, consistently oriented 2-manifold";
          return false;
        }
        e.w = c;
        out.edge_tris[it->second].y = t;
      }
    }
  }
  for (auto& e : out.edges)
    if (e.w < 0) {
      why = "mesh: open boundary edge";
      return false;
    }
  order_for_banks(out);
  out.edge_rest.resize(out.edges.size());
  for (size_t i = 0; i < out.edges.size(); ++i) {
    const int4 e = out.edges[i];
    V3 a = P(e.x), b = P(e.y), c = P(e.z), d = P(e.w);
    V3 ev = sub(b, a);
    V3 n1 = crs(ev, sub(c, a)), n2 = crs(sub(a, b), sub(d, b));
    const double L = std::sqrt(dt3(ev, ev));
    const double th = std::atan2(dt3(crs(n1, n2), ev) / L, dt3(n1, n2));
    out.edge_rest[i] = make_float4((float)L, (float)std::cos(th), (float)std::sin(th), 0.f);
  }
  out.area0.resize(nt);
  out.A0 = out.V0 = 0;
  for (int t = 0; t < nt; ++t) {
    V3 p0 = P(out.tris[t].x), p1 = P(out.tris[t].y), p2 = P(out.tris[t].z);
    V3 N = crs(sub(p1, p0), sub(p2, p0));
    const double A = 0.5 * std::sqrt(dt3(N, N));
    out.area0[t] = (float)A;
    out.A0 += A;
    out.V0 += dt3(p0, crs(p1, p2)) / 6.0;
  }
  if (!(out.V0 > 0)) {
    why = "mesh: non-positive rest volume (triangles must be counter-clockwise seen from outside)";
    return false;
  }
  // per-vertex lists of (edge, role) and (triangle, slot), CSR
  std::vector<std::vector<int>> ve(nv), vt(nv);
  for (size_t e = 0; e < out.edges.size(); ++e) {
    const int4 E = out.edges[e];
    ve[E.x].push_back((int)(e << 2) | 0);
    ve[E.y].push_back((int)(e << 2) | 1);
    ve[E.z].push_back((int)(e << 2) | 2);
    ve[E.w].push_back((int)(e << 2) | 3);
  }
  for (int t = 0; t < nt; ++t) {
    vt[out.tris[t].x].push_back((t << 2) | 0);
    vt[out.tris[t].y].push_back((t << 2) | 1);
    vt[out.tris[t].z].push_back((t << 2) | 2);
  }
  out.v_edge_start.assign(1, 0);
  out.v_tri_start.assign(1, 0);
  out.v_edge.clear();
  out.v_tri.clear();
  for (int v = 0; v < nv; ++v) {
    out.v_edge.insert(out.v_edge.end(), ve[v].begin(), ve[v].end());
    out.v_tri.insert(out.v_tri.end(), vt[v].begin(), vt[v].end());
    out.v_edge_start.push_back((int)out.v_edge.size());
    out.v_tri_start.push_back((int)out.v_tri.size());
  }
  return true;
}

template <typename T>
int upload(ibm_lbm_t* h, std::vector<Alloc>& pool, T** dst, const T* src, size_t count) {
  *dst = static_cast<T*>(dalloc(h, pool, sizeof(T) * count));
  if (!*dst) return fail(h, IBM_LBM_E_NOMEM, "device allocation failed");
  if (count) CUDA_TRY(h, cudaMemcpy(*dst, src, sizeof(T) * count, cudaMemcpyHostToDevice));
  return IBM_LBM_OK;
}

void quat_matrix(const double q[4], double R[3][3]) {
  const double w = q[0], x = q[1], y = q[2], z = q[3];
  R[0][0] = 1 - 2 * (y * y + z * z); R[0][1] = 2 * (x * y - w * z);     R[0][2] = 2 * (x * z + w * y);
  R[1][0] = 2 * (x * y + w * z);     R[1][1] = 1 - 2 * (x * x + z * z); R[1][2] = 2 * (y * z - w * x);
  R[2][0] = 2 * (x * z - w * y);     R[2][1] = 2 * (y * z + w * x);     R[2][2] = 1 - 2 * (x * x + y * y);
}

bool fluid_yz(const LatticeDev& L, int y, int z) {
  if (L.geometry == GEOM_YWALLS) return y >= 0 && y < L.ny;
  if (L.geometry == GEOM_TUBE) {
    if (y < 0 || y >= L.ny || z < 0 || z >= L.nz) return false;
    const float dy = (float)y - L.yc, dz = (float)z - L.zc;
    return !(dy * dy + dz * dz > L.R2);
  }
  return true;
}

std::vector<RowInfo> build_rows(const LatticeDev& L) {
  std::vector<RowInfo> rows;
  const int nx = L.nx, ny = L.ny, nz = L.nz;
  for (int z = 0; z < nz; ++z)
    for (int y = 0; y < ny; ++y) {
      if (!fluid_yz(L, y, z)) continue;
      RowInfo R{};
      R.base = nx * (y + ny * z);
      R.y = y;
      R.trow = L.ntx * ((y >> TILE_Y_SHIFT) + L.nty * (z >> TILE_Z_SHIFT));
      R.oyp = (y == ny - 1) ? -(ny - 1) * nx : nx;
      R.oym = (y == 0) ? (ny - 1) * nx : -nx;
      R.ozp = (z == nz - 1) ? -(nz - 1) * nx * ny : nx * ny;
      R.ozm = (z == 0) ? (nz - 1) * nx * ny : -nx * ny;
      int mask = 0;
      for (int dy = -1; dy <= 1; ++dy)
        for (int dz = -1; dz <= 1; ++dz) {
          int yy = y + dy, zz = z + dz;
          if (L.geometry == GEOM_PERIODIC) continue;
          if (L.geometry == GEOM_YWALLS) zz = (zz + nz) % nz;
          if (!fluid_yz(L, yy, zz)) mask |= 1 << ((dy + 1) * 3 + (dz + 1));
        }
      R.smask = mask;
      rows.push_back(R);
    }
  return rows;
}

// Cell-list buffers of the Morse interaction for the current markers:
// bins at least rc wide on every axis, at most morse_max_bins() of them.
int prepare_morse(ibm_lbm_t* h) {
  release_pool(h, h->morse_mem);
  h->morse_ready = false;
  const int M = h->m.M;
  const double rc = h->morse_rc;
  // neighbour lists: cutoff rc + skin, rebuilt after a move of skin / 2
  const double skin = 0.3 * rc;
  constexpr int kListCap = 48;
  const int n[3] = {h->cfg.nx, h->cfg.ny, h->cfg.nz};
  int nb[3];
  for (int a = 0; a < 3; ++a) nb[a] = std::max(1, (int)std::floor(n[a] / (rc + skin)));
  while ((long long)nb[0] * nb[1] * nb[2] > morse_max_bins()) {
    const int a = nb[0] >= nb[1] && nb[0] >= nb[2] ? 0 : (nb[1] >= nb[2] ? 1 : 2);
    nb[a] = std::max(1, nb[a] / 2);
  }
  MorseDev& P = h->morse;
  P = MorseDev{};
  P.D0 = (float)h->morse_D0;
  P.alpha = (float)h->morse_alpha;
  P.r0 = (float)h->morse_r0;
  P.rc2 = (float)(rc * rc);
  P.rl2 = (float)((rc + skin) * (rc + skin));
  P.half_skin2 = (float)(0.25 * skin * skin);
  P.cap = kListCap;
  for (int a = 0; a < 3; ++a) {
    P.nb[a] = nb[a];
    P.inv_bs[a] = (float)nb[a] / (float)n[a];
  }
  P.n_bins = nb[0] * nb[1] * nb[2];
  P.owner = h->owner;
  const size_t Mx = (size_t)std::max(M, 1);
  P.count = (int*)dalloc(h, h->morse_mem, sizeof(int) * P.n_bins);
  P.start = (int*)dalloc(h, h->morse_mem, sizeof(int) * ((size_t)P.n_bins + 1));
  P.block_sum = (int*)dalloc(h, h->morse_mem, sizeof(int) * (size_t)morse_scan_tiles(P.n_bins));
  P.bin_of = (int*)dalloc(h, h->morse_mem, sizeof(int) * Mx);
  P.rank = (int*)dalloc(h, h->morse_mem, sizeof(int) * Mx);
  P.sorted = (float4*)dalloc(h, h->morse_mem, sizeof(float4) * Mx);
  P.sorted_id = (int*)dalloc(h, h->morse_mem, sizeof(int) * Mx);
  P.bin_owner = (int*)dalloc(h, h->morse_mem, sizeof(int) * P.n_bins);
  P.ref = (float4*)dalloc(h, h->morse_mem, sizeof(float4) * Mx);
  P.cur = (float4*)dalloc(h, h->morse_mem, sizeof(float4) * Mx);
  P.n_nbr = (int*)dalloc(h, h->morse_mem, sizeof(int) * Mx);
  P.nbr = (int*)dalloc(h, h->morse_mem, sizeof(int) * Mx * kListCap);
  P.flags = (int*)dalloc(h, h->morse_mem, sizeof(int) * 2);
  if (!P.count || !P.start || !P.block_sum || !P.bin_of || !P.rank || !P.sorted || !P.sorted_id || !P.bin_owner ||
      !P.ref || !P.cur || !P.n_nbr || !P.nbr || !P.flags)
    return fail(h, IBM_LBM_E_NOMEM, "device allocation failed");
  const int flags0[2] = {1, 0};  // build the lists at the first step
  CUDA_TRY(h, cudaMemcpy(P.flags, flags0, sizeof(flags0), cudaMemcpyHostToDevice));
  CUDA_TRY(h, cudaMemset(P.ref, 0, sizeof(float4) * Mx));
  CUDA_TRY(h, cudaMemset(P.n_nbr, 0, sizeof(int) * Mx));
  CUDA_TRY(h, cudaMemset(P.count, 0, sizeof(int) * P.n_bins));
  CUDA_TRY(h, cudaMemset(P.bin_owner, 0xff, sizeof(int) * P.n_bins));
  CUDA_TRY(h, cudaMemset(P.start, 0, sizeof(int) * ((size_t)P.n_bins + 1)));
  h->morse_ready = true;
  return IBM_LBM_OK;
}

}  // namespace

bool ibm::ensure_second_buffer(ibm_lbm* h) {
  if (h->gbuf2) return true;
  const size_t bytes = sizeof(float4) * (size_t)h->L.N;
  float4* g = (float4*)dalloc(h, h->lattice_mem, bytes);
  if (!g || cudaMemsetAsync(g, 0, bytes, h->stream) != cudaSuccess) return false;  // (freed with the lattice)
  h->gbuf2 = g;
  return true;
}

extern "C" {

const char* ibm_lbm_version(void) { return "ibm_lbm 0.1 (sm_103a)"; }

const char* ibm_lbm_last_error(const ibm_lbm_t* h) {
  if (!h) return "null handle";
  return h->err.c_str();
}

void* ibm_lbm_stream(ibm_lbm_t* h) { return h ? (void*)h->stream : nullptr; }

size_t ibm_lbm_device_bytes(const ibm_lbm_t* h) { return h ? h->bytes : 0; }

static int impl_ibm_lbm_create(const ibm_lbm_config* cfg, const ibm_lbm_allocator* alloc, void* stream, ibm_lbm_t** out) {
  if (!cfg || !out) return IBM_LBM_E_ARG;
  *out = nullptr;
  const long long N = (long long)cfg->nx * cfg->ny * cfg->nz;
  if (cfg->nx < 4 || cfg->ny < 4 || cfg->nz < 4 || N >= (1LL << 31)) return IBM_LBM_E_ARG;
  if (!(cfg->tau > 0.5) || cfg->geometry < 0 || cfg->geometry > 2 || cfg->storage < 0 || cfg->storage > 2)
    return IBM_LBM_E_ARG;
  if (cfg->geometry == 2 && !(cfg->tube_radius > 0)) return IBM_LBM_E_ARG;
  if (alloc && (!alloc->alloc || !alloc->release)) return IBM_LBM_E_ARG;
  ibm_lbm_t* h = new ibm_lbm_t();
  h->cfg = *cfg;
  if (alloc) {
    h->alloc = *alloc;
    h->has_alloc = true;
  }
  auto bail = [&](int code) {
    ibm_lbm_destroy(h);
    return code;
  };
  if (cudaSetDevice(cfg->device) != cudaSuccess) {
    cudaGetLastError();
    return bail(IBM_LBM_E_CUDA);
  }
  if (stream) {
    h->stream = (cudaStream_t)stream;
  } else {
    if (cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking) != cudaSuccess) return bail(IBM_LBM_E_CUDA);
    h->own_stream = true;
  }
  LatticeDev& L = h->L;
  L.nx = cfg->nx; L.ny = cfg->ny; L.nz = cfg->nz; L.N = (int)N;
  L.geometry = cfg->geometry;
  L.omega = (float)(1.0 / cfg->tau);
  L.guo_pre = (float)(1.0 - 0.5 / cfg->tau);
  L.wall_u0 = (float)cfg->wall_u[0]; L.wall_u1 = (float)cfg->wall_u[1];
  L.yc = 0.5f * (float)(cfg->ny - 1); L.zc = 0.5f * (float)(cfg->nz - 1);
  L.R2 = (float)(cfg->tube_radius * cfg->tube_radius);
  L.g0x = (float)cfg->body_force[0]; L.g0y = (float)cfg->body_force[1]; L.g0z = (float)cfg->body_force[2];
  L.by_nx = fast_div((unsigned)cfg->nx);
  L.ntx = (cfg->nx + 31) >> TILE_X_SHIFT;
  L.nty = (cfg->ny + 3) >> TILE_Y_SHIFT;
  L.ntz = (cfg->nz + 3) >> TILE_Z_SHIFT;
  const size_t sp = cfg->storage == STORE_F32 ? 4 : 2;
  L.pop = dalloc(h, h->lattice_mem, (size_t)Q * N * sp);
  L.uw = (float4*)dalloc(h, h->lattice_mem, sizeof(float4) * N);
  h->gbuf = (float4*)dalloc(h, h->lattice_mem, sizeof(float4) * N);
  h->fbuf = (uint8_t*)dalloc(h, h->lattice_mem, (size_t)tiles(L));
  h->fbuf2 = (uint8_t*)dalloc(h, h->lattice_mem, (size_t)tiles(L));
  L.g = h->gbuf;  // every view of the lattice (steps, stages, server) carries them
  L.flags = h->fbuf;
  L.status = (int*)dalloc(h, h->lattice_mem, 256);
  h->d_diag = (double*)dalloc(h, h->lattice_mem, 8 * sizeof(double));
  h->d_umax = (unsigned*)dalloc(h, h->lattice_mem, 256);
  if (!L.pop || !L.uw || !h->gbuf || !h->fbuf || !h->fbuf2 || !L.status || !h->d_diag ||
      !h->d_umax) {
    h->err = "device allocation failed";
    return bail(IBM_LBM_E_NOMEM);
  }
  {
    std::vector<RowInfo> rows = build_rows(L);
    h->n_rows = (int)rows.size();
    if (upload<RowInfo>(h, h->lattice_mem, &h->rows, rows.data(), rows.size())) return bail(IBM_LBM_E_NOMEM);
  }
  if (cudaDeviceGetAttribute(&h->n_sm, cudaDevAttrMultiProcessorCount, cfg->device) != cudaSuccess)
    return bail(IBM_LBM_E_CUDA);
  if (transfer_configure() != cudaSuccess || couple_configure() != cudaSuccess ||
      cluster_configure() != cudaSuccess || cluster_capacity(1, &h->clusters_one) != cudaSuccess ||
      cluster_capacity(CLUSTER_PER_SM, &h->clusters_two) != cudaSuccess) {
    cudaGetLastError();
    return bail(IBM_LBM_E_CUDA);
  }
  if (cudaMallocHost((void**)&h->h_diag, 8 * sizeof(double) + 2 * sizeof(unsigned) + sizeof(int)) != cudaSuccess)
    return bail(IBM_LBM_E_NOMEM);
  h->h_umax = reinterpret_cast<unsigned*>(h->h_diag + 8);
  h->h_status = reinterpret_cast<int*>(h->h_umax + 2);
  if (cudaMemsetAsync(L.status, 0, sizeof(int), h->stream) != cudaSuccess) return bail(IBM_LBM_E_CUDA);
  int rc = ibm_lbm_set_lattice(h, nullptr, nullptr);
  if (rc) return bail(rc);
  *out = h;
  return IBM_LBM_OK;
}

static int impl_ibm_lbm_destroy(ibm_lbm_t* h) {
  if (!h) return IBM_LBM_OK;
  if (h->stream) cudaStreamSynchronize(h->stream);
  for (auto e : h->events) cudaEventDestroy(e);
  h->events.clear();
  drop_graphs(h);
  release_pool(h, h->morse_mem);
  release_pool(h, h->marker_mem);
  release_pool(h, h->lattice_mem);
  if (h->h_diag) cudaFreeHost(h->h_diag);
  if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
  delete h;
  return IBM_LBM_OK;
}

static int impl_ibm_lbm_set_lattice(ibm_lbm_t* h, const double* rho, const double* u) {
  if (!h) return IBM_LBM_E_ARG;
  LatticeDev& L = h->L;
  const size_t N = (size_t)L.N;
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  // the caller's FP64 arrays go to the device as they are and are converted
  // there (a host conversion loop over N cells costs more than the copy)
  std::vector<Alloc> tmp;
  double* d_rho = rho ? (double*)dalloc(h, tmp, sizeof(double) * N) : nullptr;
  double* d_u = u ? (double*)dalloc(h, tmp, sizeof(double) * 3 * N) : nullptr;
  if ((rho && !d_rho) || (u && !d_u)) {
    release_pool(h, tmp);
    return fail(h, IBM_LBM_E_NOMEM, "set_lattice: device allocation failed");
  }
  touch_pages(rho, sizeof(double) * N, false);
  touch_pages(u, sizeof(double) * 3 * N, false);
  int rc = IBM_LBM_OK;
  if (rho && cudaMemcpyAsync(d_rho, rho, sizeof(double) * N, cudaMemcpyHostToDevice, h->stream) != cudaSuccess)
    rc = IBM_LBM_E_CUDA;
  if (!rc && u && cudaMemcpyAsync(d_u, u, sizeof(double) * 3 * N, cudaMemcpyHostToDevice, h->stream) != cudaSuccess)
    rc = IBM_LBM_E_CUDA;
  if (!rc) {
    launch_set_moments(L, d_rho, d_u, h->stream);
    if (cudaStreamSynchronize(h->stream) != cudaSuccess) rc = IBM_LBM_E_CUDA;
  }
  release_pool(h, tmp);
  if (rc) return fail(h, rc, "set_lattice: CUDA error");
  launch_init_equilibrium(L, h->cfg.storage, h->stream);
  CUDA_TRY(h, cudaGetLastError());
  CUDA_TRY(h, cudaMemsetAsync(h->gbuf, 0, sizeof(float4) * N, h->stream));
  CUDA_TRY(h, cudaMemsetAsync(h->fbuf, 0, (size_t)tiles(L), h->stream));
  CUDA_TRY(h, cudaMemsetAsync(L.status, 0, sizeof(int), h->stream));
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  h->density_waiting = false;
  h->steps = 0;
  h->odd_next = false;
  return IBM_LBM_OK;
}

static int impl_ibm_lbm_set_populations(ibm_lbm_t* h, const double* f) {
  if (!h || !f) return fail(h, IBM_LBM_E_ARG, "null argument");
  std::vector<Alloc> tmp;
  const size_t bytes = sizeof(double) * Q * (size_t)h->L.N;
  double* d = (double*)dalloc(h, tmp, bytes);
  if (!d) return fail(h, IBM_LBM_E_NOMEM, "device allocation failed");
  int rc = IBM_LBM_OK;
  if (cudaMemcpyAsync(d, f, bytes, cudaMemcpyHostToDevice, h->stream) != cudaSuccess) rc = IBM_LBM_E_CUDA;
  if (!rc) {
    launch_import(h->L, h->cfg.storage, d, h->stream);
    if (cudaStreamSynchronize(h->stream) != cudaSuccess) rc = IBM_LBM_E_CUDA;
  }
  release_pool(h, tmp);
  if (rc) return fail(h, rc, "set_populations: CUDA error");
  // the parity restarts: clear the force density and its flags
  CUDA_TRY(h, cudaMemsetAsync(h->gbuf, 0, sizeof(float4) * (size_t)h->L.N, h->stream));
  CUDA_TRY(h, cudaMemsetAsync(h->fbuf, 0, (size_t)tiles(h->L), h->stream));
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  h->density_waiting = false;
  h->odd_next = false;
  return IBM_LBM_OK;
}

static int impl_ibm_lbm_get_populations(ibm_lbm_t* h, double* f) {
  if (!h || !f) return fail(h, IBM_LBM_E_ARG, "null argument");
  std::vector<Alloc> tmp;
  const size_t bytes = sizeof(double) * Q * (size_t)h->L.N;
  double* d = (double*)dalloc(h, tmp, bytes);
  if (!d) return fail(h, IBM_LBM_E_NOMEM, "device allocation failed");
  launch_export(h->L, h->cfg.storage, h->odd_next, d, h->stream);
  touch_pages(f, bytes, true);
  int rc = IBM_LBM_OK;
  if (cudaMemcpyAsync(f, d, bytes, cudaMemcpyDeviceToHost, h->stream) != cudaSuccess ||
      cudaStreamSynchronize(h->stream) != cudaSuccess)
    rc = IBM_LBM_E_CUDA;
  release_pool(h, tmp);
  if (rc) return fail(h, rc, "get_populations: CUDA error");
  return IBM_LBM_OK;
}

// Forget the markers, bodies, template and Morse lists (and the graphs that
// captured them): the handle is then a lattice without markers.
static void clear_markers(ibm_lbm_t* h) {
  drop_graphs(h);
  release_pool(h, h->morse_mem);
  release_pool(h, h->marker_mem);
  h->m = MarkersDev{};
  h->morse_ready = false;
  h->owner = nullptr;
  h->solid_v = nullptr;
  h->filament_list = nullptr;
  h->n_filaments = 0;
  h->n_bodies = 0;
  h->d_bodies = nullptr;
  h->h_bodies.clear();
  h->mesh = MeshDev{};
  h->membrane_list = h->rigid_list = nullptr;
  h->n_membranes = h->n_rigids = 0;
  h->groups = nullptr;
  h->n_groups = 0;
  h->n_body_groups = 0;
  h->tracers_everywhere = false;
  h->boxes = nullptr;
  h->couple_items = nullptr;
  h->n_couple = 0;
  h->couple_order = nullptr;
  h->cluster_boxes = nullptr;
  h->cluster_max = 0;
  h->need_zero_F = false;
}

// Mean cells of the box of a body's stencils, over at most 16 of the bodies
// (3 us for 812 markers).
static double mean_box(const ibm_lbm_body* bodies, int n, const double* X, int M) {
  const int taken = std::min(n, 16);
  double sum = 0.0;
  for (int i = 0; i < taken; ++i) {
    const ibm_lbm_body& B = bodies[(int64_t)i * n / taken];
    double cells = 1.0;
    for (int a = 0; a < 3; ++a) {
      const double* x = X + a * (size_t)M + B.first;
      const auto ends = std::minmax_element(x, x + B.count);
      cells *= std::floor(*ends.second) - std::floor(*ends.first) + 4.0;
    }
    sum += cells;
  }
  return sum / taken;
}

// Lattices of more cells mark packed tracers' tiles (see set_markers_into).
constexpr int PACKED_TRACERS_CELLS = 1 << 23;

// Whether tracers lie in a sixteenth of the tiles or more.
static bool tracers_scattered(const ibm_lbm_t* h, const std::vector<MarkerGroup>& groups, const double* X, int M) {
  const LatticeDev& L = h->L;
  const int n[3] = {L.nx, L.ny, L.nz}, shift[3] = {TILE_X_SHIFT, TILE_Y_SHIFT, TILE_Z_SHIFT};
  std::vector<char> seen((size_t)tiles(L), 0);
  int64_t found = 0;
  for (const MarkerGroup& G : groups)
    for (int k = G.first; k < G.first + G.count; ++k) {
      int t[3];
      for (int a = 0; a < 3; ++a) {
        const double x = X[a * (size_t)M + k];
        const int c = (int)(x - n[a] * std::floor(x / n[a]));  // in [0, n]
        t[a] = std::min(c, n[a] - 1) >> shift[a];
      }
      char& s = seen[(size_t)t[0] + (size_t)L.ntx * (t[1] + (size_t)L.nty * t[2])];
      found += !s;
      s = 1;
      if (16 * found >= (int64_t)seen.size()) return true;
    }
  return false;
}

// set_markers after the old markers are gone; on error the caller clears
// whatever this allocated, so that a failed call leaves no half-built state.
static int set_markers_into(ibm_lbm_t* h, const ibm_lbm_mesh* mesh, int32_t n_bodies, const ibm_lbm_body* bodies,
                     int64_t n_markers, const double* X) {
  const int M = (int)n_markers;
  // validate bodies
  std::vector<std::pair<int64_t, int64_t>> ranges;
  bool any_membrane = false, any_rigid = false;
  int64_t covered = 0;
  for (int b = 0; b < n_bodies; ++b) {
    const ibm_lbm_body& B = bodies[b];
    if (B.first < 0 || B.count <= 0 || B.first + B.count > n_markers)
      return fail(h, IBM_LBM_E_ARG, "set_markers: body marker range out of bounds");
    if (B.kind == IBM_LBM_BODY_MEMBRANE) {
      any_membrane = true;
      if (!mesh) return fail(h, IBM_LBM_E_ARG, "set_markers: membrane body without a mesh");
      if (B.count != mesh->n_vertices)
        return fail(h, IBM_LBM_E_ARG, "set_markers: membrane marker count != mesh vertex count");
    } else if (B.kind == IBM_LBM_BODY_RIGID || B.kind == IBM_LBM_BODY_RIGID_DIRECT) {
      any_rigid = true;
      if (!(B.mass > 0) || !(B.inertia[0] > 0) || !(B.inertia[1] > 0) || !(B.inertia[2] > 0) || !(B.kappa >= 0))
        return fail(h, IBM_LBM_E_ARG, "set_markers: rigid body needs mass, inertia > 0 and kappa >= 0");
    } else if (B.kind == IBM_LBM_BODY_FILAMENT) {
      if (B.count < 2 || !(B.l0 > 0) || !(B.kBT_p >= 0) || !(B.k_b >= 0))
        return fail(h, IBM_LBM_E_ARG, "set_markers: filament needs >= 2 beads, l0 > 0, kBT_p >= 0 and k_b >= 0");
    } else {
      return fail(h, IBM_LBM_E_ARG, "set_markers: unknown body kind");
    }
    ranges.push_back({B.first, B.first + B.count});
    covered += B.count;
  }
  std::sort(ranges.begin(), ranges.end());
  for (size_t i = 1; i < ranges.size(); ++i)
    if (ranges[i].first < ranges[i - 1].second) return fail(h, IBM_LBM_E_ARG, "set_markers: bodies overlap");
  HostMesh hm;
  if (any_membrane) {
    std::string why;
    if (!build_mesh(mesh, hm, why)) return fail(h, IBM_LBM_E_ARG, why);
    if (hm.edges.size() >= 16384 || (size_t)mesh->n_triangles >= 16384)
      return fail(h, IBM_LBM_E_ARG, "set_markers: membrane template has too many edges or triangles");
  }
  // floor(X) of every coordinate must fit the stencil cache's int32
  for (size_t i = 0; i < 3 * (size_t)M; ++i)
    if (!(std::fabs(X[i]) < 1073741824.0))
      return fail(h, IBM_LBM_E_ARG, "set_markers: positions must be finite with |X| < 2^30");
  int rc;
  // marker arrays
  h->m.M = M;
  if ((rc = upload<double>(h, h->marker_mem, &h->m.X, X, 3 * (size_t)M))) return rc;
  h->m.U = (float4*)dalloc(h, h->marker_mem, sizeof(float4) * (size_t)M);
  h->m.F = (float4*)dalloc(h, h->marker_mem, sizeof(float4) * (size_t)M);
  h->m.cell = (int*)dalloc(h, h->marker_mem, sizeof(int) * 3 * (size_t)M);
  h->m.frac = (float*)dalloc(h, h->marker_mem, sizeof(float) * 3 * (size_t)M);
  if (!h->m.U || !h->m.F || !h->m.cell || !h->m.frac) return fail(h, IBM_LBM_E_NOMEM, "device allocation failed");
  launch_stencil_cache(h->m, h->stream);
  CUDA_TRY(h, cudaGetLastError());
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  CUDA_TRY(h, cudaMemset(h->m.U, 0, sizeof(float4) * (size_t)std::max(M, 1)));
  CUDA_TRY(h, cudaMemset(h->m.F, 0, sizeof(float4) * (size_t)std::max(M, 1)));
  // rigid body-frame offsets r_k = R^T (X_k - C)
  if (any_rigid) {
    std::vector<double> ref(3 * (size_t)M, 0.0);
    for (int b = 0; b < n_bodies; ++b) {
      const ibm_lbm_body& B = bodies[b];
      if (B.kind != IBM_LBM_BODY_RIGID && B.kind != IBM_LBM_BODY_RIGID_DIRECT) continue;
      double R[3][3];
      quat_matrix(B.quat, R);
      for (int64_t k = B.first; k < B.first + B.count; ++k) {
        const double d[3] = {X[k] - B.center[0], X[M + k] - B.center[1], X[2 * (size_t)M + k] - B.center[2]};
        for (int a = 0; a < 3; ++a) ref[a * (size_t)M + k] = R[0][a] * d[0] + R[1][a] * d[1] + R[2][a] * d[2];
      }
    }
    double* dref = nullptr;
    if ((rc = upload<double>(h, h->marker_mem, &dref, ref.data(), ref.size()))) return rc;
    h->m.ref = dref;
  }
  // body table
  std::vector<BodyDev> bd(std::max(n_bodies, 1));
  for (int b = 0; b < n_bodies; ++b) {
    const ibm_lbm_body& B = bodies[b];
    BodyDev& D = bd[b];
    D.kind = B.kind;
    D.first = (int)B.first;
    D.count = (int)B.count;
    D.kBT_p = (float)B.kBT_p; D.k_b = (float)B.k_b; D.k_l = (float)B.k_l; D.k_g = (float)B.k_g; D.k_v = (float)B.k_v;
    D.kappa = B.kappa; D.mass = B.mass;
    D.inv_mass = B.mass > 0 ? 1.0 / B.mass : 0.0;
    D.l0 = (float)B.l0;
    for (int a = 0; a < 3; ++a) {
      D.inertia[a] = B.inertia[a];
      D.inv_inertia[a] = B.inertia[a] > 0 ? 1.0 / B.inertia[a] : 0.0;
      D.center[a] = B.center[a]; D.vel[a] = B.vel[a]; D.omega[a] = B.omega[a];
    }
    for (int a = 0; a < 4; ++a) D.quat[a] = B.quat[a];
    h->h_bodies.push_back(B);
  }
  if ((rc = upload<BodyDev>(h, h->marker_mem, &h->d_bodies, bd.data(), bd.size()))) return rc;
  h->n_bodies = n_bodies;
  {
    std::vector<int> mem, rig, fil;
    std::vector<int> own((size_t)std::max(M, 1), -1);
    for (int b = 0; b < n_bodies; ++b) {
      const int kind = bodies[b].kind;
      const bool rigid = kind == IBM_LBM_BODY_RIGID || kind == IBM_LBM_BODY_RIGID_DIRECT;
      (kind == IBM_LBM_BODY_MEMBRANE ? mem : rigid ? rig : fil).push_back(b);
      if (!rigid)
        for (int64_t k = bodies[b].first; k < bodies[b].first + bodies[b].count; ++k) own[k] = b;
    }
    h->n_membranes = (int)mem.size();
    h->n_rigids = (int)rig.size();
    h->n_filaments = (int)fil.size();
    if ((rc = upload<int>(h, h->marker_mem, &h->membrane_list, mem.data(), mem.size()))) return rc;
    if ((rc = upload<int>(h, h->marker_mem, &h->rigid_list, rig.data(), rig.size()))) return rc;
    if ((rc = upload<int>(h, h->marker_mem, &h->filament_list, fil.data(), fil.size()))) return rc;
    if ((rc = upload<int>(h, h->marker_mem, &h->owner, own.data(), own.size()))) return rc;
  }
  // mesh
  if (any_membrane) {
    // pack the topology into 16-byte-aligned sections of one buffer
    std::vector<unsigned char> buf;
    auto section = [&](const void* src, size_t bytes) {
      const int off = (int)buf.size();
      buf.resize(buf.size() + ((bytes + 15) / 16) * 16, 0);
      if (bytes) std::memcpy(buf.data() + off, src, bytes);
      return off;
    };
    std::vector<ushort4> e16(hm.edges.size());
    std::vector<ushort2> et16(hm.edges.size());
    for (size_t e = 0; e < hm.edges.size(); ++e) {
      e16[e] = make_ushort4(hm.edges[e].x, hm.edges[e].y, hm.edges[e].z, hm.edges[e].w);
      et16[e] = make_ushort2(hm.edge_tris[e].x, hm.edge_tris[e].y);
    }
    std::vector<ushort4> t16(hm.tris.size());
    for (size_t t = 0; t < hm.tris.size(); ++t) t16[t] = make_ushort4(hm.tris[t].x, hm.tris[t].y, hm.tris[t].z, 0);
    auto to16 = [](const std::vector<int>& v) { return std::vector<unsigned short>(v.begin(), v.end()); };
    const auto ves = to16(hm.v_edge_start), vel = to16(hm.v_edge), vts = to16(hm.v_tri_start), vtl = to16(hm.v_tri);
    MeshDev& D = h->mesh;
    D.off_edges = section(e16.data(), e16.size() * sizeof(ushort4));
    D.off_edge_tris = section(et16.data(), et16.size() * sizeof(ushort2));
    D.off_edge_rest = section(hm.edge_rest.data(), hm.edge_rest.size() * sizeof(float4));
    D.off_tris = section(t16.data(), t16.size() * sizeof(ushort4));
    D.off_area0 = section(hm.area0.data(), hm.area0.size() * sizeof(float));
    D.off_ve_start = section(ves.data(), ves.size() * 2);
    D.off_ve = section(vel.data(), vel.size() * 2);
    D.off_vt_start = section(vts.data(), vts.size() * 2);
    D.off_vt = section(vtl.data(), vtl.size() * 2);
    const size_t whole = buf.size();
    if (!h->lean &&
        h->n_membranes <= std::max(membrane_clusters_max(h, mesh->n_vertices),
                                   h->served_slots > 0 ? 0 : solid_clusters_max(h, mesh->n_vertices))) {
      // parts of consecutive vertices for the clusters (cluster_body.cuh)
      int table[CLUSTER][8] = {};
      D.part_tris = 0;
      const int per = cluster_per(mesh->n_vertices);
      for (int p = 0; p < CLUSTER; ++p) {
        const MeshPartHost P = mesh_part_of(hm, p * per, std::min(mesh->n_vertices, (p + 1) * per));
        const int t[8] = {(int)P.edges.size(), (int)P.tris.size(), P.nt_own,
                          section(P.edges.data(), P.edges.size() * sizeof(ushort4)),
                          section(P.edge_tris.data(), P.edge_tris.size() * sizeof(ushort2)),
                          section(P.edge_rest.data(), P.edge_rest.size() * sizeof(float4)),
                          section(P.tris.data(), P.tris.size() * sizeof(ushort4)),
                          section(P.area0.data(), P.area0.size() * sizeof(float))};
        std::copy(t, t + 8, table[p]);
        D.part_tris = std::max(D.part_tris, t[1]);
      }
      D.off_parts = section(table, sizeof(table));
    }
    unsigned char* dpk = nullptr;
    rc = upload<unsigned char>(h, h->marker_mem, &dpk, buf.data(), buf.size());
    if (rc == IBM_LBM_E_NOMEM && buf.size() > whole) {  // without the parts: the paths that need none
      buf.resize(whole);
      D.off_parts = D.part_tris = 0;
      rc = upload<unsigned char>(h, h->marker_mem, &dpk, buf.data(), buf.size());
    }
    if (rc) return rc;
    D.packed_bytes = (int)buf.size();
    D.packed = dpk;
    D.nv = mesh->n_vertices;
    D.nt = mesh->n_triangles;
    D.ne = (int)hm.edges.size();
    D.work_floats = (int)membrane_work_floats(D.nv, D.nt, D.ne);
    D.A0 = (float)hm.A0;
    D.V0 = (float)hm.V0;
    // the rest area and volume are about 2^20 units of the coarse half of the sums
    D.fix_a = std::ldexp(1.0f, 20 - std::ilogb(hm.A0));
    D.fix_v = std::ldexp(1.0f, 20 - std::ilogb(hm.V0));
    int most = 1;  // contributions a vertex receives: its edge roles and triangles
    for (int v = 0; v < D.nv; ++v)
      most = std::max(most, hm.v_edge_start[v + 1] - hm.v_edge_start[v] + hm.v_tri_start[v + 1] - hm.v_tri_start[v]);
    D.qcap = (float)((2147483647.0 - 4096.0) / (double)most);
    int dev = 0, optin = 0;
    CUDA_TRY(h, cudaGetDevice(&dev));
    CUDA_TRY(h, cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    if (forces_configure(D, (size_t)optin) != cudaSuccess) {
      cudaGetLastError();
      return fail(h, IBM_LBM_E_ARG, "set_markers: membrane template too large for one thread block's shared memory");
    }
  }
  // transfer groups: bodies in chunks of BODY_GROUP, tracer runs in chunks of TRACER_GROUP
  std::vector<MarkerGroup> tracer_groups;
  {
    std::vector<MarkerGroup> groups;
    std::vector<std::pair<int64_t, int>> cuts;  // (first marker, body) in marker order
    for (int b = 0; b < n_bodies; ++b) cuts.push_back({bodies[b].first, b});
    std::sort(cuts.begin(), cuts.end());
    int64_t pos = 0;
    std::vector<char> is_tracer;
    auto add_run = [&](int64_t a, int64_t b, int step, int flags) {
      for (int64_t s0 = a; s0 < b; s0 += step) {
        groups.push_back({(int)s0, (int)std::min<int64_t>(step, b - s0), flags});
        is_tracer.push_back(step == TRACER_GROUP);
      }
    };
    for (auto& c : cuts) {
      const ibm_lbm_body& B = bodies[c.second];
      add_run(pos, B.first, TRACER_GROUP, 0);
      add_run(B.first, B.first + B.count, BODY_GROUP, B.kind == IBM_LBM_BODY_RIGID_DIRECT ? GROUP_FIXED : 0);
      pos = B.first + B.count;
    }
    add_run(pos, n_markers, TRACER_GROUP, 0);
    // Transfer blocks in the order of a Morton curve through the groups'
    // mean positions (cells / 8 per axis, periodic x wrapped): blocks that
    // run close in time then work on neighbouring cells, so the overlapping
    // parts of their boxes are served from L2 rather than HBM.
    {
      const double nxd = (double)h->cfg.nx;
      auto spread_bits = [](uint32_t v) {  // 10 bits -> every third of 30
        uint64_t x = v & 0x3ffu;
        x = (x | (x << 16)) & 0x30000ffull;
        x = (x | (x << 8)) & 0x300f00full;
        x = (x | (x << 4)) & 0x30c30c3ull;
        x = (x | (x << 2)) & 0x9249249ull;
        return x;
      };
      std::vector<std::pair<uint64_t, size_t>> key(groups.size());
      for (size_t g = 0; g < groups.size(); ++g) {
        double c[3] = {0.0, 0.0, 0.0};
        for (int k = groups[g].first; k < groups[g].first + groups[g].count; ++k)
          for (int a = 0; a < 3; ++a) c[a] += X[a * (size_t)M + k];
        uint32_t q[3];
        for (int a = 0; a < 3; ++a) {
          double v = c[a] / (double)groups[g].count;
          if (a == 0) v -= nxd * std::floor(v / nxd);
          q[a] = (uint32_t)std::min(1023.0, std::max(0.0, v / 8.0));
        }
        key[g] = {spread_bits(q[0]) | (spread_bits(q[1]) << 1) | (spread_bits(q[2]) << 2), g};
      }
      std::stable_sort(key.begin(), key.end(),
                       [](const std::pair<uint64_t, size_t>& a, const std::pair<uint64_t, size_t>& b) {
                         return a.first < b.first;
                       });
      // the bodies' groups first, then the tracers'
      std::vector<MarkerGroup> ordered;
      ordered.reserve(groups.size());
      for (int tracers = 0; tracers < 2; ++tracers) {
        for (size_t g = 0; g < groups.size(); ++g)
          if (is_tracer[key[g].second] == tracers) ordered.push_back(groups[key[g].second]);
        if (!tracers) h->n_body_groups = (int)ordered.size();
      }
      groups.swap(ordered);
      tracer_groups.assign(groups.begin() + h->n_body_groups, groups.end());
      // Tracers whose blocks fill up the waves that the bodies' take anyway (a
      // block an SM while there are few) ride along instead of taking kernels of
      // their own. us a step, along / apart: 1 body of 812 markers with 100
      // tracers 67.4/71.7, 20,000 (79 blocks) 67.7/72.6, 50,000 (197) 90.4/76.6; 40
      // membranes and 5000 61.2/65.5, 50,000 81.2/70.3; 60 of each and 5000 (140)
      // 103/107, 10,000 (160) 114/107; 200 membranes and 20,000 (279) 127/132,
      // 50,000 (396) 150/137.
      const int bodies_only = h->n_body_groups, all = (int)groups.size();
      auto waves = [&](int n) { return (n + h->n_sm - 1) / h->n_sm; };
      if (bodies_only > 0 && all < LANE_MAX_GROUPS && waves(all) == waves(bodies_only)) h->n_body_groups = all;
    }
    h->n_groups = (int)groups.size();
    if ((rc = upload<MarkerGroup>(h, h->marker_mem, &h->groups, groups.data(), groups.size()))) return rc;
    // fused path: every marker belongs to a membrane whose template fits the
    // fused kernel, one transfer group per body
    bool fused = n_bodies > 0 && covered == n_markers && any_membrane && couple_fits(h->mesh);
    for (int b = 0; b < n_bodies && fused; ++b) fused = bodies[b].kind == IBM_LBM_BODY_MEMBRANE;
    // While the separate kernels have four lanes a marker (few groups), they are
    // the faster ones for large cells, whose slabs or markers one block works off
    // alone. us a step, fused / separate, 60 spheres of radius 6, 8, 10, 14 (boxes
    // of 4.5, 8.6, 14.7, 34 thousand cells): 92 vertices 33.5/34.5, 52.8/38.7,
    // 83.5/58.1, 164/94; 252 39/42, 60/52, 94/70, 201/105; 642 50/60, 75/75, 114/102,
    // 282/140; 812 54/68, 80/84, 122/121, 305/155; 250 of them with 642 116/138,
    // 181/200, 271/271, 676/479; 520 (one thread a marker) 222/233, -, 544/545, 1253/1215.
    if (fused && n_bodies < LANE_MAX_GROUPS)
      fused = mean_box(bodies, n_bodies, X, M) <= BOX_CELLS + 8.0 * h->mesh.nv;
    if (fused) {
      std::unordered_map<int, int> body_of_first;
      for (int b = 0; b < n_bodies; ++b) body_of_first[(int)bodies[b].first] = b;
      // items[g] = (body, g) for every group g in order: the fused kernel's
      // block g reads group g and its box directly
      std::vector<int2> items;
      for (size_t g = 0; g < groups.size() && fused; ++g) {
        auto it = body_of_first.find(groups[g].first);
        if (it == body_of_first.end() || groups[g].count != (int)bodies[it->second].count) fused = false;
        else items.push_back(make_int2(it->second, (int)g));
      }
      if (fused && (int)items.size() == n_bodies && items.size() == groups.size()) {
        if ((rc = upload<int2>(h, h->marker_mem, &h->couple_items, items.data(), items.size()))) return rc;
        h->couple_order = (unsigned char*)dalloc(h, h->marker_mem, couple_order_bytes(h->mesh) * items.size());
        if (!h->couple_order) return fail(h, IBM_LBM_E_NOMEM, "device allocation failed");
        h->n_couple = (int)items.size();
      }
    }
    h->boxes = (int4*)dalloc(h, h->marker_mem, sizeof(int4) * 2 * std::max<size_t>(1, groups.size()));
    if (!h->boxes) return fail(h, IBM_LBM_E_NOMEM, "device allocation failed");
    // no box until the first spreading: an interpolation run before it (the
    // stage interface allows that) takes the per-marker path
    CUDA_TRY(h, cudaMemset(h->boxes, 0, sizeof(int4) * 2 * std::max<size_t>(1, groups.size())));
  }
  // clusters: bodies of a size one cluster takes, nothing else
  if (!h->lean) {
    bool few = n_bodies > 0 && covered == n_markers && h->n_filaments == 0 &&
               h->n_membranes <= membrane_clusters_max(h, h->mesh.nv);
    int least_rigid = INT_MAX, most_rigid = 0;
    bool direct = false;
    for (int b = 0; b < n_bodies && few; ++b) {
      const int count = (int)bodies[b].count;
      few = bodies[b].count <= CLUSTER_MAX_COUNT;
      h->cluster_max = std::max(h->cluster_max, count);
      if (bodies[b].kind == IBM_LBM_BODY_MEMBRANE) continue;
      least_rigid = std::min(least_rigid, count);
      most_rigid = std::max(most_rigid, count);
      direct |= bodies[b].kind == IBM_LBM_BODY_RIGID_DIRECT;
    }
    few = few && h->n_rigids <= rigid_clusters_max(h, least_rigid, most_rigid, direct);
    // a second wave of bodies whose boxes do not fit one block's shared memory
    // loses to the separate kernels (60 of 36 x 24 x 24: 262 us a step, 254)
    if (few && h->served_slots == 0 && h->n_rigids > h->clusters_two)
      few = mean_box(bodies, n_bodies, X, M) <= BOX_CELLS;
    few = few && (h->n_rigids == 0 ||
                  cluster_box_cells(cluster_fixed_words(h->cluster_max, 0, 0), per_sm(h, h->n_rigids)) > 0);
    few = few && (h->n_membranes == 0 ||
                  (h->mesh.part_tris > 0 &&
                   cluster_box_cells(cluster_fixed_words(h->mesh.nv, h->mesh.nv, h->mesh.part_tris),
                                     per_sm(h, h->n_membranes)) > 0));
    if (few) {
      const size_t bytes = sizeof(int4) * 2 * CLUSTER * (size_t)n_bodies;
      int4* boxes = (int4*)dalloc(h, h->marker_mem, bytes);
      if (!boxes) return fail(h, IBM_LBM_E_NOMEM, "device allocation failed");
      CUDA_TRY(h, cudaMemset(boxes, 0, bytes));
      h->cluster_boxes = boxes;
    }
  }
  h->need_zero_F = covered < n_markers;
  // From a tracer per four tiles on the stencils (up to 8 tiles each) reach
  // most of them where they are scattered: marking costs more than the
  // velocities of the other cells (a 131x96x110 box with 150,000: 63 us against
  // 16 bytes of 168 per cell). Packed tracers are marked instead where those
  // velocities do not stay in L2: us a step, marked / all velocities, tracers
  // in 0, 7, 22 and 100 % of the tiles: 256^3, 20,000 of them 418/437, 426/440,
  // 438/443, 469/444; 150,000 439/451, 470/456, 478/463, 536/492; 176^3, 2904
  // 144/149, -, -, -, 150,000 170/164; 128^3, 20,000 67/66, 71/67, 77/67, 81/69.
  h->tracers_everywhere = h->n_body_groups < h->n_groups && 4 * (n_markers - covered) >= (int64_t)tiles(h->L) &&
                          (h->L.N <= PACKED_TRACERS_CELLS || tracers_scattered(h, tracer_groups, X, M));
  if (h->morse_rc > 0.0) return prepare_morse(h);
  return IBM_LBM_OK;
}

static int impl_ibm_lbm_set_markers(ibm_lbm_t* h, const ibm_lbm_mesh* mesh, int32_t n_bodies, const ibm_lbm_body* bodies,
                                    int64_t n_markers, const double* X) {
  if (!h) return IBM_LBM_E_ARG;
  if (n_bodies < 0 || n_markers < 0 || n_markers >= (1LL << 31) || (n_markers > 0 && !X) ||
      (n_bodies > 0 && !bodies))
    return fail(h, IBM_LBM_E_ARG, "set_markers: bad counts or null arrays");
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  clear_markers(h);
  const int rc = set_markers_into(h, mesh, n_bodies, bodies, n_markers, X);
  if (rc != IBM_LBM_OK) {
    const std::string why = h->err;
    clear_markers(h);
    h->err = why;
  }
  return rc;
}

static int impl_ibm_lbm_solid_steps(ibm_lbm_t* h, int64_t n_steps, double dt, double gamma, double mass, const double* f_ext) {
  if (!h) return IBM_LBM_E_ARG;
  if (n_steps < 0 || !(dt > 0.0) || !(gamma >= 0.0) || !(mass > 0.0))
    return fail(h, IBM_LBM_E_ARG, "solid_steps: needs n_steps >= 0, dt > 0, gamma >= 0, mass > 0");
  if (h->n_rigids > 0) return fail(h, IBM_LBM_E_STATE, "solid_steps: rigid bodies need the fluid");
  const size_t M = (size_t)h->m.M;
  if (M == 0 || n_steps == 0) return IBM_LBM_OK;
  cudaStream_t st = h->stream;
  CUDA_TRY(h, cudaStreamSynchronize(st));
  if (h->need_zero_F) CUDA_TRY(h, cudaMemsetAsync(h->m.F, 0, sizeof(float4) * M, st));
  if (!h->solid_v) {
    h->solid_v = (double*)dalloc(h, h->marker_mem, sizeof(double) * 3 * M);
    if (!h->solid_v) return fail(h, IBM_LBM_E_NOMEM, "device allocation failed");
    CUDA_TRY(h, cudaMemset(h->solid_v, 0, sizeof(double) * 3 * M));
  }
  std::vector<Alloc> tmp;
  double* fe = nullptr;
  if (f_ext) {
    fe = (double*)dalloc(h, tmp, sizeof(double) * 3 * M);
    if (!fe) return fail(h, IBM_LBM_E_NOMEM, "device allocation failed");
    if (cudaMemcpy(fe, f_ext, sizeof(double) * 3 * M, cudaMemcpyHostToDevice) != cudaSuccess) {
      release_pool(h, tmp);
      return fail(h, IBM_LBM_E_CUDA, "solid_steps: copy of f_ext failed");
    }
  }
  // Few membranes and nothing else: a cluster per body, SOLID_CHUNK steps a
  // launch (a few ms).
  const bool clusters = h->n_membranes > 0 && h->n_membranes == h->n_bodies && !h->need_zero_F &&
                        !(h->morse_rc > 0.0) && h->n_membranes <= solid_clusters_max(h, h->mesh.nv) &&
                        h->mesh.part_tris > 0 && solid_cluster_fits(h->mesh);
  if (clusters) {
    for (int64_t s = 0; s < n_steps; s += SOLID_CHUNK)
      launch_solid_cluster(h->m, h->d_bodies, h->membrane_list, h->n_membranes, h->mesh, h->solid_v, fe, dt, gamma,
                           mass, (int)std::min<int64_t>(SOLID_CHUNK, n_steps - s), st);
  } else {
    for (int64_t s = 0; s < n_steps; ++s) {
      // (from the second step on the forces are those the last one ended with)
      if (s == 0) enqueue_forces(h, st);
      launch_solid_half(h->m, h->solid_v, fe, dt, gamma, mass, true, st);
      enqueue_forces(h, st);
      launch_solid_half(h->m, h->solid_v, fe, dt, gamma, mass, false, st);
    }
  }
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  release_pool(h, tmp);
  if (e != cudaSuccess) return fail(h, IBM_LBM_E_CUDA, std::string("solid_steps: ") + cudaGetErrorString(e));
  return IBM_LBM_OK;
}

static int impl_ibm_lbm_set_morse(ibm_lbm_t* h, double D0, double alpha, double r0, double rc) {
  if (!h) return IBM_LBM_E_ARG;
  if (rc > 0.0 && (!(D0 >= 0.0) || !(alpha > 0.0) || !std::isfinite(r0) || !std::isfinite(rc)))
    return fail(h, IBM_LBM_E_ARG, "set_morse: needs D0 >= 0, alpha > 0 and finite r0, rc");
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  drop_graphs(h);
  h->morse_D0 = D0;
  h->morse_alpha = alpha;
  h->morse_r0 = r0;
  h->morse_rc = rc > 0.0 ? rc : 0.0;
  release_pool(h, h->morse_mem);
  h->morse_ready = false;
  if (h->morse_rc > 0.0 && h->owner) return prepare_morse(h);
  return IBM_LBM_OK;
}

static int impl_ibm_lbm_step_async(ibm_lbm_t* h, int64_t n_steps) {
  if (!h) return IBM_LBM_E_ARG;
  return enqueue_steps(h, n_steps);
}

static int impl_ibm_lbm_synchronize(ibm_lbm_t* h) {
  if (!h) return IBM_LBM_E_ARG;
  return finish_diagnostics(h);
}

static int impl_ibm_lbm_step(ibm_lbm_t* h, int64_t n_steps) {
  if (!h) return IBM_LBM_E_ARG;
  int rc = enqueue_steps(h, n_steps);
  if (rc) return rc;
  return finish_diagnostics(h);
}

static int impl_ibm_lbm_run_stage(ibm_lbm_t* h, int32_t stage) {
  if (!h) return IBM_LBM_E_ARG;
  cudaStream_t st = h->stream;
  // The interpolation gathers from the stencil boxes the last spreading
  // computed; they hold the markers only while no stage has moved them since
  // (the interpolation advects, the direct rigid forcing places markers).
  // Otherwise the boxes are cleared first and every marker takes the
  // per-marker path.
  switch (stage) {
    case IBM_LBM_STAGE_FORCES:
      if (h->need_zero_F) CUDA_TRY(h, cudaMemsetAsync(h->m.F, 0, sizeof(float4) * (size_t)h->m.M, st));
      enqueue_forces(h, st);
      h->boxes_valid = false;
      break;
    case IBM_LBM_STAGE_SPREAD: {
      const LatticeDev L = h->L;
      CUDA_TRY(h, cudaMemsetAsync(L.flags, 0, (size_t)tiles(L), st));
      launch_spread(L, h->m, h->groups, h->n_groups, h->boxes, st);
      h->boxes_valid = true;
      h->density_waiting = true;
      break;
    }
    case IBM_LBM_STAGE_COLLIDE:
      launch_collide(h->L, h->rows, h->n_rows, h->cfg.storage, h->odd_next, true, false, st);
      h->odd_next = !h->odd_next;
      break;
    case IBM_LBM_STAGE_INTERP:
      if (!h->boxes_valid && h->n_groups > 0)
        CUDA_TRY(h, cudaMemsetAsync(h->boxes, 0, sizeof(int4) * 2 * (size_t)h->n_groups, st));
      launch_interpolate(h->L, h->m, h->groups, h->n_groups, h->boxes, st);
      h->boxes_valid = false;
      h->density_waiting = false;
      h->steps += 1;
      break;
    default:
      return fail(h, IBM_LBM_E_ARG, "unknown stage");
  }
  CUDA_TRY(h, cudaGetLastError());
  CUDA_TRY(h, cudaStreamSynchronize(st));
  return IBM_LBM_OK;
}

static int impl_ibm_lbm_set_marker_forces(ibm_lbm_t* h, const double* F) {
  if (!h || (!F && h->m.M > 0)) return fail(h, IBM_LBM_E_ARG, "null argument");
  const size_t M = (size_t)h->m.M;
  std::vector<float4> tmp(M);
  for (size_t k = 0; k < M; ++k) tmp[k] = make_float4((float)F[k], (float)F[M + k], (float)F[2 * M + k], 0.f);
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  if (M) CUDA_TRY(h, cudaMemcpy(h->m.F, tmp.data(), sizeof(float4) * M, cudaMemcpyHostToDevice));
  return IBM_LBM_OK;
}

static int impl_ibm_lbm_get_force_density(ibm_lbm_t* h, double* g) {
  if (!h || !g) return fail(h, IBM_LBM_E_ARG, "null argument");
  const size_t N = (size_t)h->L.N;
  std::vector<float4> tmp(N);
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  CUDA_TRY(h, cudaMemcpy(tmp.data(), h->gbuf, sizeof(float4) * N, cudaMemcpyDeviceToHost));
  for (size_t i = 0; i < N; ++i) {
    g[i] = tmp[i].x; g[N + i] = tmp[i].y; g[2 * N + i] = tmp[i].z;
  }
  return IBM_LBM_OK;
}

static int impl_ibm_lbm_get_fields(ibm_lbm_t* h, double* rho, double* u) {
  if (!h) return IBM_LBM_E_ARG;
  const LatticeDev& L = h->L;
  const size_t N = (size_t)L.N;
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  if (!rho && !u) return IBM_LBM_OK;
  // expanded to the FP64 layout on the device, then one copy per array
  std::vector<Alloc> tmp;
  double* d_rho = rho ? (double*)dalloc(h, tmp, sizeof(double) * N) : nullptr;
  double* d_u = u ? (double*)dalloc(h, tmp, sizeof(double) * 3 * N) : nullptr;
  if ((rho && !d_rho) || (u && !d_u)) {
    release_pool(h, tmp);
    return fail(h, IBM_LBM_E_NOMEM, "get_fields: device allocation failed");
  }
  launch_get_moments(L, d_rho, d_u, h->stream);
  // while the kernel runs: take the page faults of freshly allocated output
  // arrays on several threads (the copy would take them one by one)
  touch_pages(rho, sizeof(double) * N, true);
  touch_pages(u, sizeof(double) * 3 * N, true);
  int rc = IBM_LBM_OK;
  if (rho && cudaMemcpyAsync(rho, d_rho, sizeof(double) * N, cudaMemcpyDeviceToHost, h->stream) != cudaSuccess)
    rc = IBM_LBM_E_CUDA;
  if (!rc && u && cudaMemcpyAsync(u, d_u, sizeof(double) * 3 * N, cudaMemcpyDeviceToHost, h->stream) != cudaSuccess)
    rc = IBM_LBM_E_CUDA;
  if (cudaStreamSynchronize(h->stream) != cudaSuccess) rc = IBM_LBM_E_CUDA;
  release_pool(h, tmp);
  if (rc) return fail(h, rc, "get_fields: CUDA error");
  return IBM_LBM_OK;
}

static int impl_ibm_lbm_get_markers(ibm_lbm_t* h, double* X, double* U, double* F) {
  if (!h) return IBM_LBM_E_ARG;
  const size_t M = (size_t)h->m.M;
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  if (M == 0) return IBM_LBM_OK;
  // U and F expanded to the FP64 [3][M] layout on the device
  std::vector<Alloc> tmp;
  double* dU = U ? (double*)dalloc(h, tmp, sizeof(double) * 3 * M) : nullptr;
  double* dF = F ? (double*)dalloc(h, tmp, sizeof(double) * 3 * M) : nullptr;
  if ((U && !dU) || (F && !dF)) {
    release_pool(h, tmp);
    return fail(h, IBM_LBM_E_NOMEM, "get_markers: device allocation failed");
  }
  if (U) launch_expand_xyz(h->m.U, dU, (int)M, h->stream);
  if (F) launch_expand_xyz(h->m.F, dF, (int)M, h->stream);
  touch_pages(X, sizeof(double) * 3 * M, true);
  touch_pages(U, sizeof(double) * 3 * M, true);
  touch_pages(F, sizeof(double) * 3 * M, true);
  int rc = IBM_LBM_OK;
  if (X && cudaMemcpyAsync(X, h->m.X, sizeof(double) * 3 * M, cudaMemcpyDeviceToHost, h->stream) != cudaSuccess)
    rc = IBM_LBM_E_CUDA;
  if (!rc && U && cudaMemcpyAsync(U, dU, sizeof(double) * 3 * M, cudaMemcpyDeviceToHost, h->stream) != cudaSuccess)
    rc = IBM_LBM_E_CUDA;
  if (!rc && F && cudaMemcpyAsync(F, dF, sizeof(double) * 3 * M, cudaMemcpyDeviceToHost, h->stream) != cudaSuccess)
    rc = IBM_LBM_E_CUDA;
  if (cudaStreamSynchronize(h->stream) != cudaSuccess) rc = IBM_LBM_E_CUDA;
  release_pool(h, tmp);
  if (rc) return fail(h, rc, "get_markers: CUDA error");
  return IBM_LBM_OK;
}

static int impl_ibm_lbm_get_bodies(ibm_lbm_t* h, ibm_lbm_body* bodies, int32_t n_bodies) {
  if (!h || n_bodies != h->n_bodies || (n_bodies > 0 && !bodies))
    return fail(h, IBM_LBM_E_ARG, "get_bodies: count mismatch");
  if (n_bodies == 0) return IBM_LBM_OK;
  std::vector<BodyDev> bd(n_bodies);
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  CUDA_TRY(h, cudaMemcpy(bd.data(), h->d_bodies, sizeof(BodyDev) * n_bodies, cudaMemcpyDeviceToHost));
  for (int b = 0; b < n_bodies; ++b) {
    ibm_lbm_body B = h->h_bodies[b];
    for (int a = 0; a < 3; ++a) {
      B.center[a] = bd[b].center[a]; B.vel[a] = bd[b].vel[a]; B.omega[a] = bd[b].omega[a];
    }
    for (int a = 0; a < 4; ++a) B.quat[a] = bd[b].quat[a];
    bodies[b] = B;
  }
  return IBM_LBM_OK;
}

static int impl_ibm_lbm_set_timing(ibm_lbm_t* h, int64_t max_steps) {
  if (!h || max_steps < 0 || max_steps > (1 << 22)) return fail(h, IBM_LBM_E_ARG, "set_timing: bad step count");
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  for (auto e : h->events) cudaEventDestroy(e);
  h->events.clear();
  h->timed_steps = 0;
  h->timed_odd.clear();
  h->timed_fused.clear();
  h->timing = max_steps > 0;
  for (int64_t i = 0; i < 5 * max_steps; ++i) {
    cudaEvent_t e;
    CUDA_TRY(h, cudaEventCreate(&e));
    h->events.push_back(e);
  }
  return IBM_LBM_OK;
}

static int impl_ibm_lbm_set_timing_fused(ibm_lbm_t* h, int on) {
  if (!h) return IBM_LBM_E_ARG;
  h->timing_fused = on != 0;
  return IBM_LBM_OK;
}

static int impl_ibm_lbm_get_timing(ibm_lbm_t* h, double out[6]) {
  if (!h || !out) return IBM_LBM_E_ARG;
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  for (int k = 0; k < 6; ++k) out[k] = 0.0;
  for (size_t s = 0; s < h->timed_steps; ++s)
    for (int k = h->timed_fused[s] ? 2 : 0; k < 4; ++k) {
      float ms = 0.f;
      CUDA_TRY(h, cudaEventElapsedTime(&ms, h->events[5 * s + k], h->events[5 * s + k + 1]));
      out[k] += ms;
      if (k == 2 && h->timed_odd[s]) out[5] += ms;
    }
  out[4] = (double)h->timed_steps;
  h->timed_steps = 0;
  h->timed_odd.clear();
  h->timed_fused.clear();
  return IBM_LBM_OK;
}

static int impl_ibm_lbm_get_diagnostics(ibm_lbm_t* h, double out[8]) {
  if (!h || !out) return IBM_LBM_E_ARG;
  int rc = enqueue_diagnostics(h);
  if (rc) return rc;
  CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  h->diag_pending = false;
  float umax2;
  std::memcpy(&umax2, h->h_umax, sizeof(float));
  out[0] = h->h_diag[4] + h->h_diag[0];
  out[1] = h->h_diag[1];
  out[2] = h->h_diag[2];
  out[3] = h->h_diag[3];
  out[4] = std::sqrt((double)umax2);
  out[5] = (double)h->steps;
  out[6] = h->h_diag[4];
  out[7] = 0.0;
  return IBM_LBM_OK;
}


int ibm_lbm_create(const ibm_lbm_config* cfg, const ibm_lbm_allocator* alloc, void* stream, ibm_lbm_t** out) {
  return abi_guard(nullptr, [&]() -> int { return impl_ibm_lbm_create(cfg, alloc, stream, out); });
}

int ibm_lbm_destroy(ibm_lbm_t* h) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_destroy(h); });
}

int ibm_lbm_set_lattice(ibm_lbm_t* h, const double* rho, const double* u) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_set_lattice(h, rho, u); });
}

int ibm_lbm_set_populations(ibm_lbm_t* h, const double* f) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_set_populations(h, f); });
}

int ibm_lbm_get_populations(ibm_lbm_t* h, double* f) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_get_populations(h, f); });
}

int ibm_lbm_set_markers(ibm_lbm_t* h, const ibm_lbm_mesh* mesh, int32_t n_bodies, const ibm_lbm_body* bodies,
                        int64_t n_markers, const double* X) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_set_markers(h, mesh, n_bodies, bodies, n_markers, X); });
}

int ibm_lbm_solid_steps(ibm_lbm_t* h, int64_t n_steps, double dt, double gamma, double mass, const double* f_ext) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_solid_steps(h, n_steps, dt, gamma, mass, f_ext); });
}

int ibm_lbm_set_morse(ibm_lbm_t* h, double D0, double alpha, double r0, double rc) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_set_morse(h, D0, alpha, r0, rc); });
}

int ibm_lbm_step_async(ibm_lbm_t* h, int64_t n_steps) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_step_async(h, n_steps); });
}

int ibm_lbm_synchronize(ibm_lbm_t* h) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_synchronize(h); });
}

int ibm_lbm_step(ibm_lbm_t* h, int64_t n_steps) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_step(h, n_steps); });
}

int ibm_lbm_run_stage(ibm_lbm_t* h, int32_t stage) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_run_stage(h, stage); });
}

int ibm_lbm_set_marker_forces(ibm_lbm_t* h, const double* F) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_set_marker_forces(h, F); });
}

int ibm_lbm_get_force_density(ibm_lbm_t* h, double* g) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_get_force_density(h, g); });
}

int ibm_lbm_get_fields(ibm_lbm_t* h, double* rho, double* u) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_get_fields(h, rho, u); });
}

int ibm_lbm_get_markers(ibm_lbm_t* h, double* X, double* U, double* F) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_get_markers(h, X, U, F); });
}

int ibm_lbm_get_bodies(ibm_lbm_t* h, ibm_lbm_body* bodies, int32_t n_bodies) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_get_bodies(h, bodies, n_bodies); });
}

int ibm_lbm_set_timing(ibm_lbm_t* h, int64_t max_steps) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_set_timing(h, max_steps); });
}

int ibm_lbm_set_timing_fused(ibm_lbm_t* h, int on) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_set_timing_fused(h, on); });
}

int ibm_lbm_get_timing(ibm_lbm_t* h, double out[6]) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_get_timing(h, out); });
}

int ibm_lbm_get_diagnostics(ibm_lbm_t* h, double out[8]) {
  return abi_guard(h, [&]() -> int { return impl_ibm_lbm_get_diagnostics(h, out); });
}
}  // extern "C"
