// lbm_runtime.cu -- host runtime behind the C ABI of include/lbm.h: handle
// state, device memory (library-owned or caller-bound), stream, CUDA-graph
// replay of the step loop, the three step forms (bulk + NSBC kernel pair,
// fused one-launch kernel, staged producer/consumer kernel) in their plain
// or far-field-shifted variant, launch-shape autotuning, and the entry
// points.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <type_traits>
#include <mutex>
#include <string>
#include <vector>

#include "lbm.h"
#include "lbm_aux.cuh"
#include "lbm_kernels.cuh"
#include "lbm_multistep.cuh"
#include "lbm_staged.cuh"
#include "lbm_trace.h"
#include "lbm_tune_cache.h"

namespace lbmk {
Shift<double> far_field_shift(const double m0[3]) {
  Shift<double> z{};
  const double drho = m0[0] - 1.0, rho = m0[0], ux = m0[1], uy = m0[2];
  const double usq = 1.5 * (ux * ux + uy * uy);
  for (int i = 0; i < 9; ++i) {
    const double cu = cx(i) * ux + cy(i) * uy;
    z.sh[i] = wt<double>(i) * (drho + rho * (3.0 * cu + 4.5 * cu * cu - usq));
  }
  for (int i = 0; i < 9; ++i) {
    const double cu = cx(i) * ux + cy(i) * uy;
    z.p0[i] = 1.0 + 3.0 * cu + 4.5 * cu * cu - usq;
  }
  z.u0[0] = ux;
  z.u0[1] = uy;
  z.rho0 = rho;
  for (int c = 0; c < 3; ++c) z.m0[c] = m0[c];
  z.on = !(drho == 0.0 && ux == 0.0 && uy == 0.0);
  return z;
}
}  // namespace lbmk

namespace {

thread_local std::string g_last_error;

int fail(int code, const char* fmt, ...) __attribute__((format(printf, 2, 3)));
int fail(int code, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  g_last_error = buf;
  return code;
}

}  // namespace

// Shared with the other translation units of the library (batched mode):
// records the calling thread's error message and returns `code`.
int lbm_internal_fail(int code, const char* msg) {
  g_last_error = msg;
  return code;
}

namespace {

#define LBM_CUDA(call)                                                                          \
  do {                                                                                          \
    cudaError_t e_ = (call);                                                                    \
    if (e_ != cudaSuccess)                                                                      \
      return fail(e_ == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA, "%s: %s (%s:%d)", #call, \
                  cudaGetErrorString(e_), __FILE__, __LINE__);                                  \
  } while (0)

constexpr int kGraphSteps = 16;  // steps per captured graph (even: buffers return to their roles)
constexpr int kReduceThreads = 256;
constexpr int kReduceBlocks = 1216;  // 8 x 152 SMs
constexpr int kNsbcThreads = 128;
// where pick_form() draws the lines
constexpr long long kPassNodes32 = 1200000, kPassNodes16 = 2800000, kTileNodes = 110000, kFusedNodes = 800000;
constexpr long long kTileNodesEdge = 32000, kTileNodesEdge16 = 20000;
constexpr long long kResidentNodesPeriodic = 5000, kResidentNodesAxis = 45000, kResidentNodesAxisMrt = 25000;
constexpr int kPassRows32 = 80, kPassRows16 = 320;
constexpr long long kTileCells = 1 << 21;  // largest domain the autotuner tries as tiles
// steps of a launch of the resident kernel: below, the flags' clearing and the
// cooperative launch (about 20 us together, against 0.4 us saved per step)
// outweigh what it saves; the upper bound keeps a launch to some 20 ms
constexpr int kResidentMin = 64, kResidentMax = 4096;

// How lbm_step launches steps, where it does not keep the domain resident: the bulk and NSBC kernel pair, both in one
// launch, the staged kernel, the multi-step pass, or tiles.
enum class Form { Pair = LBM_FORM_PAIR, Fused = LBM_FORM_FUSED, Staged = LBM_FORM_STAGED, Pass = LBM_FORM_PASS,
                  Tiles = LBM_FORM_TILES };

// launch shapes compiled for the bulk kernel: threads per block along x
constexpr int kShapesBX[] = {64, 128, 256, 512};
constexpr int kShapesRows[] = {1, 2, 4, 8};
// L2 prefetch distances (rows ahead) tried by the autotuner
constexpr int kPrefetchRows[] = {0, 1, 3, 8};

}  // namespace

struct lbm {
  int nx = 0, ny = 0, pitch = 0;
  long long plane = 0;  // elements per population plane (256-byte multiple)
  double tau = 0.0;
  lbmk::Nsbc nsbc{};
  int storage = LBM_F32;
  size_t elt = 4;
  void* buf[2] = {nullptr, nullptr};
  void* scratch = nullptr;
  bool owns_memory = false;
  bool bound = false;
  bool initialised = false;
  int cur = 0;  // buffer holding the current state
  long long steps = 0;
  cudaStream_t stream = nullptr;
  cudaStream_t cap = nullptr, side = nullptr;  // capture stream and NSBC branch
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
  cudaEvent_t ev_chunk[8] = {};  // row chunks of the host transfers (lbm_init, lbm_get_macros)
  cudaGraphExec_t graph[2] = {nullptr, nullptr};  // by starting buffer
  int bx = 128, rows = 1, pf = 0;  // bulk launch shape and L2 prefetch distance (rows)
  int device = 0;
  int collision = 0;                          // 0 = BGK, 1 = MRT
  double s_e = 1.0, s_eps = 1.0, s_q = 1.0;   // MRT energy, energy-square and flux rates
  // staged step kernel (lbm_set_staged): the producer/consumer kernel of
  // lbm_staged.cuh over this domain's one-instance work list; 0 = off, else
  // the number of tile stages
  int staged = 0;
  // fused step kernel (lbm_set_fused): the bulk grid of the current shape and
  // the NSBC quads in one launch per step
  bool fused = false;
  // multi-step pass (lbm_set_twostep): several steps per launch, the steps in
  // between kept on chip; the rolling items' strips, bands, rows per band,
  // bands per wave, waves and persistent grid, and the device's SM count
  bool twostep = false;
  int ts_strips = 0, ts_bands = 0, ts_band = 0, ts_wave_bands = 0, ts_waves = 0, ts_grid = 0, sms = 0;
  // tiles (lbm_set_tiles; small domains): several steps per launch of tile_kernel
  bool tiles = false;
  int tl_gx = 0, tl_gy = 0, tl_steps = 0, tl_smem = 0;
  // the domain as resident tiles (resident_kernel): halo 0 where it does not fit
  int rs_gx = 0, rs_gy = 0, rs_halo = 0, rs_smem = 0;
  // no launch form was asked for: lbm_step takes the one pick_form() names
  bool form_auto = true;
  Form form = Form::Pair;  // what prepare_form() settled on
  bool form_ready = false, rs_ready = false, tail_ready = false;
  // work counters and the resident tiles' flags: the library's own memory, as
  // bound scratch areas may be shared by handles or hold the caller's data
  // between two calls
  int* d_sync = nullptr;
  int sync_slot = -1;
  bool moved = false;  // to another stream, with a state
  bool waited = false;            // steps since the state was set hold bounded waits
  unsigned wait_limit = (unsigned)lbmk::kTmaWaitCycles;  // of the resident tiles (lbm_set_wait_limit)
  int4* d_items = nullptr;
  lbmk::InstDev* d_inst = nullptr;
  void* d_shift = nullptr;  // the far field's storage shift in the compute type (staged kernel)
  int n_items = 0, items_storage = -1, staged_grid = 0;
  // per-launch timing (lbm_profile): an event pair around every launch, and
  // which kernel it was (0 = bulk or staged step kernel, 1 = NSBC)
  bool profiling = false;
  std::vector<cudaEvent_t> ev_pool;
  std::vector<int> ev_kind;
  size_t ev_used = 0;
};

namespace {

size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

lbmk::Geom geom(const lbm_t* h) { return lbmk::Geom{h->nx, h->ny, h->pitch, h->plane}; }

size_t macro_bytes(const lbm_t* h) { return round_up((size_t)h->nx * h->ny * sizeof(double), 256); }

// scratch layout: rho | ux | uy (each macro_bytes) | partials | out[5]
double* scratch_field(lbm_t* h, int c) {
  return reinterpret_cast<double*>(static_cast<char*>(h->scratch) + c * macro_bytes(h));
}
double* scratch_partials(lbm_t* h) { return scratch_field(h, 3); }
double* scratch_out(lbm_t* h) { return scratch_partials(h) + kReduceBlocks * 4; }
// d_sync: work counter, warps or blocks done and give-up flag of the kernels
// that claim work, then the flags of the resident tiles, one per block.  A
// handle's area is a slot of an array that the library holds on each device
// (344 KB), as an allocation would cost a new handle's first steps 90 us; more
// handles than slots have one allocated.  The address is looked up each time:
// it does not survive a reset of the device.  What an earlier owner left in a
// slot is cleared with the first state.
constexpr size_t kSyncFlags = 256;
constexpr int kResidentBlocks = 160, kSyncSlots = 64, kSyncDevices = 64;
constexpr size_t kSyncBytes = kSyncFlags + (size_t)kResidentBlocks * lbmk::kFlagStride * sizeof(unsigned);
static __device__ __align__(256) unsigned char g_sync_area[kSyncSlots * kSyncBytes];
std::mutex g_sync_mutex;
uint64_t g_sync_used[kSyncDevices] = {};
static_assert(kSyncSlots == 64 && kSyncBytes % 256 == 0, "a bit per slot");

int take_sync(lbm_t* h) {
  if (h->d_sync) return LBM_OK;
  if (h->device >= 0 && h->device < kSyncDevices) {
    void* base = nullptr;
    LBM_CUDA(cudaGetSymbolAddress(&base, g_sync_area));
    std::lock_guard<std::mutex> lock(g_sync_mutex);
    uint64_t& used = g_sync_used[h->device];
    for (int k = 0; k < kSyncSlots; ++k)
      if (!(used >> k & 1)) {
        used |= 1ull << k;
        h->sync_slot = k;
        h->d_sync = reinterpret_cast<int*>(static_cast<char*>(base) + k * kSyncBytes);
        return LBM_OK;
      }
  }
  LBM_CUDA(cudaMalloc(&h->d_sync, kSyncBytes));
  return LBM_OK;
}

// (the handle's streams have been waited for)
void give_sync(lbm_t* h) {
  if (h->sync_slot >= 0) {
    std::lock_guard<std::mutex> lock(g_sync_mutex);
    g_sync_used[h->device] &= ~(1ull << h->sync_slot);
  } else if (h->d_sync) {
    cudaFree(h->d_sync);
  }
  h->sync_slot = -1;
  h->d_sync = nullptr;
}

int* sched(const lbm_t* h) { return h->d_sync; }
unsigned* resident_flags(const lbm_t* h) {
  return reinterpret_cast<unsigned*>(reinterpret_cast<char*>(h->d_sync) + kSyncFlags);
}

void drop_graphs(lbm_t* h) {
  for (auto& g : h->graph)
    if (g) {
      cudaGraphExecDestroy(g);
      g = nullptr;
    }
  h->staged_grid = 0;  // the staged kernel's residency may have changed too
  h->form_ready = false;
}

int ensure_memory(lbm_t* h) {
  if (h->bound) return LBM_OK;
  const size_t bb = lbm_buffer_bytes(h), sb = lbm_scratch_bytes(h);
  LBM_CUDA(cudaGetDevice(&h->device));
  if (int rc = take_sync(h)) return rc;
  LBM_CUDA(cudaMalloc(&h->buf[0], bb));
  LBM_CUDA(cudaMalloc(&h->buf[1], bb));
  LBM_CUDA(cudaMalloc(&h->scratch, sb));
  LBM_CUDA(cudaMemset(h->buf[0], 0, bb));
  LBM_CUDA(cudaMemset(h->buf[1], 0, bb));
  lbmk::check_add(h->buf[0], bb);  // bounds-checked build only
  lbmk::check_add(h->buf[1], bb);
  h->owns_memory = true;
  h->bound = true;
  return LBM_OK;
}

// A new state starts from clear work counters and a clear give-up flag, in
// stream order (lbm_init*: init_kernel does it).
int clear_sched(lbm_t* h) {
  LBM_CUDA(cudaMemsetAsync(sched(h), 0, 4 * sizeof(int), h->stream));
  h->waited = false;
  return LBM_OK;
}

// The end of a call that waits for the stream: LBM_ETIMEOUT if a wait of the
// steps before gave up, the state then not being one.
int sync_checked(lbm_t* h, cudaStream_t s, const char* who) {
  int flag = 0;
  if (h->waited) LBM_CUDA(cudaMemcpyAsync(&flag, sched(h) + 2, sizeof(int), cudaMemcpyDeviceToHost, s));
  LBM_CUDA(cudaStreamSynchronize(s));
  if (flag) return fail(LBM_ETIMEOUT, "%s: a bounded wait of a step kernel gave up", who);
  return LBM_OK;
}

int ensure_streams(lbm_t* h) {
  if (!h->cap) {
    LBM_CUDA(cudaStreamCreateWithFlags(&h->cap, cudaStreamNonBlocking));
    LBM_CUDA(cudaStreamCreateWithFlags(&h->side, cudaStreamNonBlocking));
    LBM_CUDA(cudaEventCreateWithFlags(&h->ev_fork, cudaEventDisableTiming));
    LBM_CUDA(cudaEventCreateWithFlags(&h->ev_join, cudaEventDisableTiming));
    for (auto& e : h->ev_chunk) LBM_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
  }
  return LBM_OK;
}

int grid_for(long long n, int threads) {
  long long b = (n + threads - 1) / threads;
  return (int)(b < 1 ? 1 : (b > 152LL * 32 ? 152LL * 32 : b));
}

// ---- typed launchers ------------------------------------------------------


// storage shift of the handle's far field (stored populations are
// deviations from its equilibrium)
lbmk::Shift<double> zshift(const lbm_t* h) { return lbmk::far_field_shift(h->nsbc.m0); }

template <typename C>
lbmk::Rates<C> rates(const lbm_t* h) {
  return lbmk::Rates<C>{C(1.0 / h->tau), C(h->s_e), C(h->s_eps), C(h->s_q), lbmk::shift_as<C>(zshift(h))};
}

// SHIFT: the far field is not at rest, so the stored populations are
// deviations from its equilibrium (Shift); the plain kernels otherwise.
template <typename F>
void with_shift(const lbm_t* h, F&& f) {
  if (zshift(h).on)
    f(std::integral_constant<bool, true>{});
  else
    f(std::integral_constant<bool, false>{});
}

template <typename T, int BX>
void launch_bulk_bx(const lbm_t* h, const void* a, void* b, int rows, cudaStream_t s) {
  using C = typename lbmk::Store<T>::C;
  constexpr int V = lbmk::Store<T>::V;
  const int nvec = (h->nx + V - 1) / V;
  dim3 grid((nvec + BX - 1) / BX, (h->ny - 2 + rows - 1) / rows);
  with_shift(h, [&](auto zc) {
    constexpr bool Z = decltype(zc)::value;
    constexpr bool PF = !std::is_same<T, float>::value || Z;  // without the prefetch: f32 at rest
    if (h->collision == 1)
      lbmk::bulk_kernel<T, BX, 1, Z><<<grid, BX, 0, s>>>(static_cast<const T*>(a), static_cast<T*>(b), geom(h),
                                                        rates<C>(h), rows, h->pf);
    else if (h->pf == 0)
      lbmk::bulk_kernel<T, BX, 0, Z, PF><<<grid, BX, 0, s>>>(static_cast<const T*>(a), static_cast<T*>(b), geom(h),
                                                            rates<C>(h), rows, 0);
    else
      lbmk::bulk_kernel<T, BX, 0, Z><<<grid, BX, 0, s>>>(static_cast<const T*>(a), static_cast<T*>(b), geom(h),
                                                        rates<C>(h), rows, h->pf);
  });
}

template <typename T>
void launch_bulk(const lbm_t* h, const void* a, void* b, int bx, int rows, cudaStream_t s) {
  switch (bx) {
    case 64: launch_bulk_bx<T, 64>(h, a, b, rows, s); break;
    case 256: launch_bulk_bx<T, 256>(h, a, b, rows, s); break;
    case 512: launch_bulk_bx<T, 512>(h, a, b, rows, s); break;
    default: launch_bulk_bx<T, 128>(h, a, b, rows, s); break;
  }
}

template <typename T>
void launch_nsbc(const lbm_t* h, const void* a, void* b, cudaStream_t s) {
  using C = typename lbmk::Store<T>::C;
  const long long perim = 2LL * h->nx + 2LL * (h->ny - 2);
  const int blocks = (int)((perim * 4 + kNsbcThreads - 1) / kNsbcThreads);
  with_shift(h, [&](auto zc) {
    constexpr bool Z = decltype(zc)::value;
    if (h->collision == 1)
      lbmk::nsbc_kernel<T, 1, Z><<<blocks, kNsbcThreads, 0, s>>>(static_cast<const T*>(a), static_cast<T*>(b),
                                                                 geom(h), h->nsbc, rates<C>(h));
    else
      lbmk::nsbc_kernel<T, 0, Z><<<blocks, kNsbcThreads, 0, s>>>(static_cast<const T*>(a), static_cast<T*>(b),
                                                                 geom(h), h->nsbc, rates<C>(h));
  });
}

template <typename T, int BX>
void launch_fused_bx(const lbm_t* h, const void* a, void* b, int rows, cudaStream_t s) {
  using C = typename lbmk::Store<T>::C;
  constexpr int V = lbmk::Store<T>::V;
  const int nvec = (h->nx + V - 1) / V;
  const int nbx = (nvec + BX - 1) / BX, nby = (h->ny - 2 + rows - 1) / rows;
  const long long perim = 2LL * h->nx + 2LL * (h->ny - 2);
  const int n_edge = (int)((perim * 4 + BX - 1) / BX);
  const int grid = n_edge + nbx * nby;
  with_shift(h, [&](auto zc) {
    constexpr bool Z = decltype(zc)::value;
    if (h->collision == 1)
      lbmk::fused_step_kernel<T, BX, 1, Z><<<grid, BX, 0, s>>>(static_cast<const T*>(a), static_cast<T*>(b), geom(h),
                                                              h->nsbc, rates<C>(h), rows, h->pf, n_edge, nbx);
    else
      lbmk::fused_step_kernel<T, BX, 0, Z><<<grid, BX, 0, s>>>(static_cast<const T*>(a), static_cast<T*>(b), geom(h),
                                                              h->nsbc, rates<C>(h), rows, h->pf, n_edge, nbx);
  });
}

// (picked by lbm_step itself: blocks of 64, which spread the boundary's quads
// over twice as many SMs -- 200^2 f64 10.6 against 13.5 us a step, 400^2 f32
// 3.6 against 3.9)
template <typename T>
void launch_fused(const lbm_t* h, const void* a, void* b, cudaStream_t s) {
  switch (h->form_auto ? 64 : h->bx) {
    case 64: launch_fused_bx<T, 64>(h, a, b, h->form_auto ? 1 : h->rows, s); break;
    case 256: launch_fused_bx<T, 256>(h, a, b, h->rows, s); break;
    case 512: launch_fused_bx<T, 512>(h, a, b, h->rows, s); break;
    default: launch_fused_bx<T, 128>(h, a, b, h->rows, s); break;
  }
}

// ---- staged step kernel --------------------------------------------------
// One launch per step: the producer warp of each block claims the domain's
// work items (NSBC chunks of 32 nodes and tiles of 128 vectors of the
// flattened interior, padding columns included) and stages the tiles into
// shared memory; the 128 consumer threads collide them.  Same device
// functions as the bulk and NSBC kernels, so the same bits.
constexpr int kStagedThreads = 128, kStagedTile = 128;

template <typename T, int MODEL, int STAGES>
const void* staged_kernel(bool shift) {
  return shift ? (const void*)lbmk::batch_ws_kernel<T, kStagedThreads, MODEL, kStagedTile, STAGES, 1, true>
               : (const void*)lbmk::batch_ws_kernel<T, kStagedThreads, MODEL, kStagedTile, STAGES, 1, false>;
}

template <typename T>
const void* staged_kernel_for(const lbm_t* h) {
  const bool z = zshift(h).on;
  if (h->staged >= 4) return h->collision == 1 ? staged_kernel<T, 1, 4>(z) : staged_kernel<T, 0, 4>(z);
  return h->collision == 1 ? staged_kernel<T, 1, 3>(z) : staged_kernel<T, 0, 3>(z);
}

int staged_smem(const lbm_t* h) { return (h->staged >= 4 ? 4 : 3) * 9 * (kStagedTile + 2) * 16; }

template <typename T>
void launch_staged(const lbm_t* h, const void* a, void* b, cudaStream_t s) {
  const T* A = static_cast<const T*>(a);
  T* B = static_cast<T*>(b);
  const int smem = staged_smem(h);
  const dim3 grid(h->staged_grid), block(kStagedThreads + 32);
  auto go = [&](auto kernel) {
    kernel<<<grid, block, smem, s>>>(A, B, h->d_inst,
                                     static_cast<const lbmk::Shift<typename lbmk::Store<T>::C>*>(h->d_shift),
                                     h->d_items, h->n_items, h->nsbc, h->s_e, h->s_eps, h->s_q, sched(h));
  };
  with_shift(h, [&](auto zc) {
    constexpr bool Z = decltype(zc)::value;
    if (h->staged >= 4) {
      if (h->collision == 1)
        go(lbmk::batch_ws_kernel<T, kStagedThreads, 1, kStagedTile, 4, 1, Z>);
      else
        go(lbmk::batch_ws_kernel<T, kStagedThreads, 0, kStagedTile, 4, 1, Z>);
    } else {
      if (h->collision == 1)
        go(lbmk::batch_ws_kernel<T, kStagedThreads, 1, kStagedTile, 3, 1, Z>);
      else
        go(lbmk::batch_ws_kernel<T, kStagedThreads, 0, kStagedTile, 3, 1, Z>);
    }
  });
}

// Multi-step pass: the rolling items are strips of Roll::OUT output columns
// times bands of rows, taken after the frame's tiles by a persistent grid of
// as many blocks as fit on the device at once; each wave of items is all
// strips of ts_wave_bands bands.
template <typename T>
void pass_grid(lbm_t* h, int per_sm) {
  using R = lbmk::Roll<T>;
  const int rows = std::max(1, h->ny - 4);  // of the shortest pass (two steps)
  h->ts_strips = (std::max(h->nx - 4, 1) + R::OUT - 1) / R::OUT;
  const int warps = std::max(1, per_sm * h->sms * R::WARPS);
  const int per_wave = std::max(1, warps / h->ts_strips);  // bands side by side
  // rows per band, 24 / 48 / 64 / 96 / 128 at 8192^2: f32 267 / 242 / 237 / 238 / 247 us a step,
  // f16 299 / 270 / 263 / 258 / 255 (4096^2 alike): a restart costs the rows above the band
  // (2 K of them), a long band the lines neighbouring strips share
  int want = sizeof(T) == 4 ? 64 : 96;
  const int waves = std::max(1, (rows + per_wave * want / 2) / (per_wave * want));
  h->ts_band = std::max(4, (rows + per_wave * waves - 1) / (per_wave * waves));
  h->ts_bands = (rows + h->ts_band - 1) / h->ts_band;
  h->ts_wave_bands = std::min(per_wave, h->ts_bands);
  h->ts_waves = (h->ts_bands + h->ts_wave_bands - 1) / h->ts_wave_bands;
  h->ts_grid = std::max(1, per_sm * h->sms);
}

template <typename T>
void launch_pass(const lbm_t* h, const void* a, void* b, int steps, cudaStream_t s) {
  using C = typename lbmk::Store<T>::C;
  const T* A = static_cast<const T*>(a);
  T* B = static_cast<T*>(b);
  const int n_tiles = lbmk::frame_tiles(h->nx, h->ny);
  with_shift(h, [&](auto zc) {
    constexpr bool Z = decltype(zc)::value;
    auto go = [&](auto kernel) {
      kernel<<<h->ts_grid, lbmk::kRollThreads, lbmk::Roll<T>::kSmem, s>>>(
          A, B, geom(h), h->nsbc, rates<C>(h), steps, n_tiles, h->ts_strips, h->ts_band, h->ts_bands,
          h->ts_wave_bands, h->ts_waves, sched(h));
    };
    if (h->collision == 1)
      go(lbmk::pass_kernel<T, 1, Z>);
    else
      go(lbmk::pass_kernel<T, 0, Z>);
  });
}

// the multi-step pass serves this handle (f32 / f16 / bf16, no periodic axis, 8 x 8 nodes or more)
bool pass_ok(const lbm_t* h) {
  return h->storage != LBM_F64 && !h->nsbc.periodic_x && !h->nsbc.periodic_y && h->nx >= 2 * lbmk::kPassSteps &&
         h->ny >= 2 * lbmk::kPassSteps;
}

template <typename T>
int pass_prepare(lbm_t* h) {
  const int smem = (int)lbmk::Roll<T>::kSmem;
  cudaError_t e = cudaSuccess;
  int per_sm = 0;
  for (const void* k : {(const void*)lbmk::pass_kernel<T, 0, false>, (const void*)lbmk::pass_kernel<T, 0, true>,
                        (const void*)lbmk::pass_kernel<T, 1, false>, (const void*)lbmk::pass_kernel<T, 1, true>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, lbmk::pass_kernel<T, 1, true>, lbmk::kRollThreads,
                                                      smem);
  if (e != cudaSuccess)
    return fail(LBM_ECUDA, "multi-step pass: %d bytes of shared memory refused: %s", smem, cudaGetErrorString(e));
  if (per_sm <= 0) return fail(LBM_ECUDA, "multi-step pass: no block fits on an SM");
  pass_grid<T>(h, per_sm);
  return LBM_OK;
}

// ---- tiles of a small domain -----------------------------------------------
// tiles serve this handle at all (every form of it is covered: storage,
// collision, edges); false for domains too narrow to cut
bool tiles_ok(const lbm_t* h) { return h->nx >= 8 && h->ny >= 8; }

template <typename T>
void launch_tiles(const lbm_t* h, const void* a, void* b, int steps, cudaStream_t s) {
  using C = typename lbmk::Store<T>::C;
  with_shift(h, [&](auto zc) {
    constexpr bool Z = decltype(zc)::value;
    auto go = [&](auto kernel) {
      kernel<<<h->tl_gx * h->tl_gy, lbmk::kTileThreads, h->tl_smem, s>>>(static_cast<const T*>(a), static_cast<T*>(b),
                                                                        geom(h), h->nsbc, rates<C>(h), h->tl_gx,
                                                                        h->tl_gy, steps);
    };
    if (h->collision == 1)
      go(lbmk::tile_kernel<T, 1, Z>);
    else
      go(lbmk::tile_kernel<T, 0, Z>);
  });
}

lbmk::TilePlan tile_plan(const lbm_t* h) {
  return lbmk::plan_tiles(h->nx, h->ny, h->storage == LBM_F64, h->nsbc.periodic_x, h->nsbc.periodic_y, h->sms);
}

template <typename T>
int tiles_prepare(lbm_t* h) {
  const lbmk::TilePlan p = tile_plan(h);
  h->tl_steps = 0;
  if (p.steps == 0) return LBM_OK;
  h->tl_gx = p.gx;
  h->tl_gy = p.gy;
  h->tl_steps = p.steps;
  h->tl_smem = p.smem;
  cudaError_t e = cudaSuccess;
  with_shift(h, [&](auto zc) {
    constexpr bool Z = decltype(zc)::value;
    const void* k = h->collision == 1 ? (const void*)lbmk::tile_kernel<T, 1, Z> : (const void*)lbmk::tile_kernel<T, 0, Z>;
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lbmk::kTileRoom);
  });
  if (e != cudaSuccess)
    return fail(LBM_ECUDA, "tiles: %d bytes of shared memory refused: %s", (int)lbmk::kTileRoom, cudaGetErrorString(e));
  return LBM_OK;
}

template <typename F>
void dispatch(int storage, F&& f) {
  switch (storage) {
    case LBM_F64: f(double{}); break;
    case LBM_F16: f(__half{}); break;
    case LBM_BF16: f(__nv_bfloat16{}); break;
    default: f(float{}); break;
  }
}

// Work list, instance record and counters of the staged kernel (built once
// the storage is fixed), and its grid: one resident wave of blocks.  Never
// called inside a stream capture (lbm_step prepares it before capturing).
int ensure_staged(lbm_t* h) {
  if (!h->staged) return LBM_OK;
  if (h->items_storage != h->storage) {
    const int V = (int)(16 / h->elt);
    lbmk::InstDev d{};
    d.off = 0;
    d.plane = h->plane;
    d.nx = h->nx;
    d.ny = h->ny;
    d.pitch = h->pitch;
    d.omega = 1.0 / h->tau;
    for (int c = 0; c < 3; ++c) d.m0[c] = h->nsbc.m0[c];
    lbmk::set_row_divisor(d, V);
    std::vector<int4> items;
    lbmk::staged_instance_items(0, d, V, kStagedTile, kStagedThreads / 4, items);
    if (h->d_items) cudaFree(h->d_items);
    h->d_items = nullptr;
    LBM_CUDA(cudaMalloc(&h->d_items, items.size() * sizeof(int4)));
    LBM_CUDA(cudaMemcpy(h->d_items, items.data(), items.size() * sizeof(int4), cudaMemcpyHostToDevice));
    if (!h->d_inst) LBM_CUDA(cudaMalloc(&h->d_inst, sizeof(lbmk::InstDev)));
    LBM_CUDA(cudaMemcpy(h->d_inst, &d, sizeof d, cudaMemcpyHostToDevice));
    if (!h->d_shift) LBM_CUDA(cudaMalloc(&h->d_shift, sizeof(lbmk::Shift<double>)));
    int rcz = LBM_OK;
    dispatch(h->storage, [&](auto tag) {
      using C = typename lbmk::Store<decltype(tag)>::C;
      const lbmk::Shift<C> z = lbmk::shift_as<C>(zshift(h));
      if (cudaMemcpy(h->d_shift, &z, sizeof z, cudaMemcpyHostToDevice) != cudaSuccess) rcz = LBM_ECUDA;
    });
    if (rcz) return fail(rcz, "staged step kernel: shift copy failed");
    h->n_items = (int)items.size();
    h->items_storage = h->storage;
  }
  if (h->staged_grid <= 0) {
    int per_sm = 0, sms = 0;
    LBM_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device));
    dispatch(h->storage, [&](auto tag) {
      using T = decltype(tag);
      const void* k = staged_kernel_for<T>(h);
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, staged_smem(h));
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kStagedThreads + 32, staged_smem(h));
    });
    if (per_sm <= 0) return fail(LBM_ECUDA, "staged step kernel: no block fits on an SM");
    h->staged_grid = std::min(h->n_items, per_sm * sms);
  }
  return LBM_OK;
}

// Equilibrium initialisation of rows [y0, y1) of both buffers (the other
// buffer's padding columns start defined too) from device fields [ny][nx].
void enqueue_init_rows(const lbm_t* h, const double* d_rho, const double* d_ux, const double* d_uy, int y0, int y1) {
  dispatch(h->storage, [&](auto tag) {
    using T = decltype(tag);
    lbmk::init_kernel<T><<<lbmk::rows_grid(h->pitch, y1 - y0), 256, 0, h->stream>>>(
        static_cast<T*>(h->buf[0]), static_cast<T*>(h->buf[1]), geom(h), zshift(h), d_rho, d_ux, d_uy, y0, y1,
        y0 == 0 ? sched(h) : nullptr);
  });
}

void enqueue_macros_rows(const lbm_t* h, double* d_rho, double* d_ux, double* d_uy, int y0, int y1) {
  dispatch(h->storage, [&](auto tag) {
    using T = decltype(tag);
    lbmk::macros_kernel<T><<<lbmk::rows_grid(h->nx, y1 - y0), 256, 0, h->stream>>>(
        static_cast<const T*>(h->buf[h->cur]), geom(h), lbmk::shift_as<typename lbmk::Store<T>::C>(zshift(h)), d_rho,
        d_ux, d_uy, y0, y1);
  });
}

// ---- a domain that stays on chip for many steps ------------------------------
template <typename T>
const void* resident_kernel_for(const lbm_t* h) {
  const void* k = nullptr;
  with_shift(h, [&](auto zc) {
    constexpr bool Z = decltype(zc)::value;
    k = h->collision == 1 ? (const void*)lbmk::resident_kernel<T, 1, Z> : (const void*)lbmk::resident_kernel<T, 0, Z>;
  });
  return k;
}

template <typename T>
int resident_prepare(lbm_t* h) {
  int coop = 0;
  LBM_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, h->device));
  if (!coop) return LBM_OK;
  const lbmk::TilePlan p = lbmk::plan_resident(h->nx, h->ny, h->nsbc.periodic_x, h->nsbc.periodic_y,
                                               std::min(h->sms, kResidentBlocks));
  if (p.steps == 0) return LBM_OK;
  cudaError_t e = cudaSuccess;
  int per_sm = 0;
  const void* k = resident_kernel_for<T>(h);
  e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lbmk::kTileRoom);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, lbmk::kTileThreads, p.smem);
  if (e != cudaSuccess)
    return fail(LBM_ECUDA, "resident tiles: %d bytes of shared memory refused: %s", p.smem, cudaGetErrorString(e));
  if (per_sm < 1) return LBM_OK;
  h->rs_gx = p.gx;
  h->rs_gy = p.gy;
  h->rs_halo = p.steps;
  h->rs_smem = p.smem;
  return LBM_OK;
}

// `steps` steps in one launch, from buffer `from`; the state is then in buffer
// from ^ (rounds & 1).  The blocks wait for one another: a cooperative launch,
// which starts all of them or none.  Their flags are zeroed before each launch.
template <typename T>
cudaError_t launch_resident(lbm_t* h, int from, int steps, cudaStream_t s) {
  using C = typename lbmk::Store<T>::C;
  T *A = static_cast<T*>(h->buf[from]), *B = static_cast<T*>(h->buf[1 - from]);
  lbmk::Geom g = geom(h);
  lbmk::Nsbc p = h->nsbc;
  lbmk::Rates<C> r = rates<C>(h);
  int gx = h->rs_gx, gy = h->rs_gy, halo = h->rs_halo;
  unsigned* flags = resident_flags(h);
  unsigned limit = h->wait_limit;
  int* err = sched(h);
  cudaError_t e =
      cudaMemsetAsync(flags, 0, (size_t)gx * gy * lbmk::kFlagStride * sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  void* args[] = {&A, &B, &g, &p, &r, &gx, &gy, &halo, &steps, &flags, &limit, &err};
  return cudaLaunchCooperativeKernel(resident_kernel_for<T>(h), dim3(gx * gy), dim3(lbmk::kTileThreads), args,
                                     h->rs_smem, s);
}

// Where the launch is refused -- a stream that may use too few SMs for all
// blocks at once -- the domain is not kept resident any more (rs_halo = 0)
// until the form is settled anew, and the caller takes the steps otherwise.
int enqueue_resident(lbm_t* h, int steps) {
  cudaError_t e = cudaSuccess;
  dispatch(h->storage, [&](auto tag) {
    using T = decltype(tag);
    if constexpr (!std::is_same<T, double>::value) e = launch_resident<T>(h, h->cur, steps, h->stream);
  });
  if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
    cudaGetLastError();
    h->rs_halo = 0;
    return LBM_OK;
  }
  if (e != cudaSuccess) return fail(LBM_ECUDA, "resident tiles: launch failed: %s", cudaGetErrorString(e));
  h->waited = true;
  h->cur ^= (steps + h->rs_halo - 1) / h->rs_halo & 1;
  return LBM_OK;
}

// A domain several times wider than high: rows are where the forms of one step
// are at their best and tiles at their worst; and the other way round.
bool wide(const lbm_t* h) { return h->nx > 4 * h->ny; }
bool tall(const lbm_t* h) { return h->ny > 4 * h->nx; }
bool thin_f32(const lbm_t* h) {
  return h->storage == LBM_F32 && h->nx < 64 && (long long)h->nx * h->ny > kTileNodes;
}

// Tiles as lbm_step's own choice, against one launch per step.  Tiles compute
// the nodes on both lines of a periodic axis with the boundary's quads and
// twice, and hold 16-bit states as floats.  Microseconds a step, tiles / one
// launch:
//   open, f32     320^2 2.91 / 2.95  2000 x 50 2.9 / 2.7   6000 x 16 3.7 / 2.8
//   open, f16     128^2 2.5 / 2.6    200^2 2.9 / 2.6       320^2 3.7 / 3.1
//   one axis      f32 160^2 2.4 / 2.5, 200^2 2.7 / 2.6     f16 160^2 2.9 / 2.7
//   both axes     f32 16^2 2.4 / 2.0, 64^2 2.2 / 2.1, 200^2 3.0 / 2.3
//   tall          f16 100 x 1000 3.6 / 4.2, 8 x 13000 8.7 / 31
bool tiles_serve(const lbm_t* h) {
  if (h->storage == LBM_F64 || !tiles_ok(h) || wide(h)) return false;
  const int axes = (h->nsbc.periodic_x != 0) + (h->nsbc.periodic_y != 0);
  const long long most = axes == 2   ? 0
                         : tall(h)   ? kTileNodes
                         : h->elt == 2 ? (axes ? kTileNodesEdge16 : kTileNodesEdge)
                                       : (axes ? kTileNodesEdge : kTileNodes);
  return (long long)h->nx * h->ny <= most;
}

// The launch form lbm_step takes when none was asked for, by size and storage
// (microseconds per step on a GB300, BGK):
//   nodes            200^2   300^2   400^2   600^2  1024^2  1200^2  1700^2  2048^2  4096^2
//   f32   one launch  3.1     3.3     3.6     5.7     9.0    14.2    33.4    46.1     181
//         tiles       2.3     2.8     3.8     6.6    14.4
//         pass                        5.2     7.2     9.8    11.3    15.8    19.0      65
//   f16   one launch                  4.0     5.6     7.4    11.0    19.8    28.5     107
//         pass                        6.8     7.5    11.5    14.3    19.2    23.6      75
// A pass is a chain of rows, so it needs enough of them to fill the chip; a
// tile's halo grows with the steps it takes.  The frame of a pass costs a node
// of the perimeter about 40 times an inner one in f32 (a pass / the pair:
// 65536 x 20 33 / 18, x 48 42 / 40, x 96 57 / 74, 20000 x 64 15.8 / 12.8,
// x 100 17.4 / 21.6), more in 16 bits (65536 x 96 62 / 46, x 160 76 / 70,
// 20000 x 250 35 / 33, 5000 x 600 18.5 / 19.5): wide domains of few rows do
// without.  Narrow ones of many rows do not: the pair's rows are short there
// (20 x 65536 f32 43 / 115), and below 64 columns one launch loses to the pair
// as well where there are enough rows (one launch / the pair, 4 x 40000: f32
// 57 / 46; in f64 and 16 bits it wins, 377 / 418 and 90 / 93).
Form pick_form(const lbm_t* h) {
  const long long nodes = (long long)h->nx * h->ny;
  const bool f32 = h->elt == 4;
  if (pass_ok(h) && nodes >= (f32 ? kPassNodes32 : kPassNodes16) &&
      (h->ny >= (f32 ? kPassRows32 : kPassRows16) || h->ny >= h->nx))
    return Form::Pass;
  if (tiles_serve(h)) return Form::Tiles;
  return nodes <= kFusedNodes && !thin_f32(h) ? Form::Fused : Form::Pair;
}

// The domain resident as lbm_step's own choice (calls of kResidentMin steps or
// more), against one launch per step; microseconds a step, resident / one
// launch:
//   open, BGK at rest   620^2 f32 4.9 / 5.0   613 x 377 f16 3.4 / 3.7   1200 x 300 f16 4.6 / 4.0
//   open, otherwise     320^2 MRT f32 3.25 / 3.26, 400^2 3.6 / 3.4   1000 x 100 3.3 / 3.0
//   one periodic axis   200^2 f32 2.54 / 2.56, bf16 2.3 / 2.7, 240^2 2.7 / 2.6; MRT 160^2 3.0 / 2.9, 200^2 3.2 / 2.9
//   both                64^2 1.8 / 2.1, MRT 2.1 / 2.2; 128^2 2.2 / 2.1, MRT 2.7 / 2.2
bool resident_serves(const lbm_t* h) {
  const long long nodes = (long long)h->nx * h->ny;
  const bool plain = h->collision == 0 && !zshift(h).on;
  const int axes = (h->nsbc.periodic_x != 0) + (h->nsbc.periodic_y != 0);
  if (axes)
    return nodes <= (axes == 2 ? kResidentNodesPeriodic : h->collision == 0 ? kResidentNodesAxis : kResidentNodesAxisMrt);
  return nodes <= (wide(h) && !plain ? kTileNodesEdge : kTileNodes) || (plain && !wide(h));
}

int device_sms(lbm_t* h) {
  if (h->sms) return LBM_OK;
  int sms = 0;
  LBM_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device));
  h->sms = sms;
  return LBM_OK;
}

// The form of the next steps, its grid and its kernels' attributes (nothing
// is allocated).
int prepare_form(lbm_t* h) {
  if (h->form_ready) return LBM_OK;
  if (int rc = device_sms(h)) return rc;
  h->form = h->form_auto             ? pick_form(h)
            : h->staged                ? Form::Staged
            : h->fused                 ? Form::Fused
            : h->twostep && pass_ok(h) ? Form::Pass
            : h->tiles && tiles_ok(h)  ? Form::Tiles
                                       : Form::Pair;
  int rc = LBM_OK;
  if (h->form == Form::Pass || h->form == Form::Tiles)
    dispatch(h->storage, [&](auto tag) {
      using T = decltype(tag);
      if (h->form == Form::Tiles) {
        rc = tiles_prepare<T>(h);
        if (h->tl_steps == 0) h->form = Form::Pair;  // the edges were changed since lbm_set_tiles: no tiling serves these
      } else if constexpr (!std::is_same<T, double>::value) {
        rc = pass_prepare<T>(h);
      }
    });
  h->rs_halo = 0;
  h->rs_ready = false;
  h->tail_ready = h->form == Form::Tiles;
  h->form_ready = rc == LBM_OK;
  return rc;
}

// The steps that the graphs of a small domain's one-launch form leave over go
// out as tiles where there are three or more: launched one by one they take
// the host 4 us each (calls of five steps, us a step, tiles / one launch: f16
// 300^2 4.1 / 5.9, 100 x 1000 4.1 / 6.2; of three 5.0 / 5.8 and 5.5 / 6.2, f32
// 223 x 43 3.4 / 4.2; of two, f16 300^2 6.2 / 5.9).
constexpr int kTailSteps = 3;
bool tail_serves(const lbm_t* h) {
  const long long nodes = (long long)h->nx * h->ny;
  return h->form_auto && h->form == Form::Fused && h->storage != LBM_F64 && tiles_ok(h) &&
         nodes <= (wide(h) ? kTileNodesEdge : kTileNodes);
}
int prepare_tail(lbm_t* h) {
  if (h->tail_ready) return LBM_OK;
  int rc = LBM_OK;
  dispatch(h->storage, [&](auto tag) { rc = tiles_prepare<decltype(tag)>(h); });
  h->tail_ready = rc == LBM_OK;
  return rc;
}

// Whether the domain can stay resident (rs_halo); settled after the form, when
// a call first has steps enough for it.
int prepare_resident(lbm_t* h) {
  if (h->rs_ready) return LBM_OK;
  int rc = LBM_OK;
  if (h->storage != LBM_F64 && tiles_ok(h) &&
      (h->form_auto ? h->form != Form::Pass && resident_serves(h) : h->form == Form::Tiles))
    dispatch(h->storage, [&](auto tag) {
      using T = decltype(tag);
      if constexpr (!std::is_same<T, double>::value) rc = resident_prepare<T>(h);
    });
  h->rs_ready = rc == LBM_OK;
  return rc;
}

int steps_per_launch(const lbm_t* h) {
  return h->form == Form::Pass ? lbmk::kPassSteps : (h->form == Form::Tiles ? h->tl_steps : 1);
}

// One step from buffer `from` to 1 - from.  With `fork`, the NSBC kernel runs
// on the side stream concurrently with the bulk kernel (both only read
// buffer `from` and write disjoint nodes of the other buffer).
void enqueue_step(const lbm_t* h, int from, cudaStream_t s, bool fork);

// One launch of `steps` steps (the form's own number or fewer) from buffer
// `from` to 1 - from; the forms of one step take one.
// tail: as tiles, whatever the form.
void enqueue_launch(const lbm_t* h, int from, int steps, cudaStream_t s, bool fork, bool tail) {
  if (tail || h->form == Form::Tiles || (h->form == Form::Pass && steps > 1)) {
    dispatch(h->storage, [&](auto tag) {
      using T = decltype(tag);
      if (tail || h->form == Form::Tiles) {
        launch_tiles<T>(h, h->buf[from], h->buf[1 - from], steps, s);
      } else if constexpr (!std::is_same<T, double>::value) {
        launch_pass<T>(h, h->buf[from], h->buf[1 - from], steps, s);
      }
    });
  } else {
    enqueue_step(h, from, s, fork);
  }
}

void enqueue_step(const lbm_t* h, int from, cudaStream_t s, bool fork) {
  const void* a = h->buf[from];
  void* b = h->buf[1 - from];
  dispatch(h->storage, [&](auto tag) {
    using T = decltype(tag);
    if (h->staged) {
      launch_staged<T>(h, a, b, s);
      return;
    }
    // (a step that no graph overlaps: one launch instead of the pair's two in
    // a row, 9.2 against about 12 us at 1024^2 f32)
    if (h->form == Form::Fused || (h->form == Form::Pair && h->form_auto && !fork && !thin_f32(h))) {
      launch_fused<T>(h, a, b, s);
      return;
    }
    if (fork) {
      cudaEventRecord(h->ev_fork, s);
      cudaStreamWaitEvent(h->side, h->ev_fork, 0);
      launch_nsbc<T>(h, a, b, h->side);
      launch_bulk<T>(h, a, b, h->bx, h->rows, s);
      cudaEventRecord(h->ev_join, h->side);
      cudaStreamWaitEvent(s, h->ev_join, 0);
    } else {
      launch_bulk<T>(h, a, b, h->bx, h->rows, s);
      launch_nsbc<T>(h, a, b, s);
    }
  });
}

int capture_graph(lbm_t* h, int from) {
  cudaGraph_t g = nullptr;
  LBM_CUDA(cudaStreamBeginCapture(h->cap, cudaStreamCaptureModeThreadLocal));
  for (int k = 0; k < kGraphSteps; ++k) enqueue_step(h, (from + k) & 1, h->cap, true);
  cudaError_t e = cudaStreamEndCapture(h->cap, &g);
  if (e != cudaSuccess) return fail(LBM_ECUDA, "graph capture failed: %s", cudaGetErrorString(e));
  e = cudaGraphInstantiate(&h->graph[from], g, 0);
  cudaGraphDestroy(g);
  if (e != cudaSuccess) return fail(LBM_ECUDA, "graph instantiate failed: %s", cudaGetErrorString(e));
  return LBM_OK;
}

// Event pair for one profiled launch of kernel `kind` (0 bulk / staged, 1 NSBC).
int profiled_pair(lbm_t* h, int kind, cudaEvent_t* e) {
  for (int k = 0; k < 2; ++k) {
    if (h->ev_used == h->ev_pool.size()) {
      cudaEvent_t x;
      LBM_CUDA(cudaEventCreate(&x));
      h->ev_pool.push_back(x);
      h->ev_kind.push_back(0);
    }
    h->ev_kind[h->ev_used] = kind;
    e[k] = h->ev_pool[h->ev_used++];
  }
  return LBM_OK;
}

// One step with an event pair around each kernel, all on the handle's stream.
int enqueue_step_profiled(lbm_t* h, int from) {
  const void* a = h->buf[from];
  void* b = h->buf[1 - from];
  cudaEvent_t e[4];
  const bool one = h->staged || h->form == Form::Fused;  // one launch per step
  int rc = profiled_pair(h, 0, e);
  if (!rc && !one) rc = profiled_pair(h, 1, e + 2);
  if (rc) return rc;
  dispatch(h->storage, [&](auto tag) {
    using T = decltype(tag);
    cudaEventRecord(e[0], h->stream);
    if (h->staged)
      launch_staged<T>(h, a, b, h->stream);
    else if (one)
      launch_fused<T>(h, a, b, h->stream);
    else
      launch_bulk<T>(h, a, b, h->bx, h->rows, h->stream);
    cudaEventRecord(e[1], h->stream);
    if (!one) {
      cudaEventRecord(e[2], h->stream);
      launch_nsbc<T>(h, a, b, h->stream);
      cudaEventRecord(e[3], h->stream);
    }
  });
  return LBM_OK;
}

// A launch of several steps with an event pair around it (counted as one bulk
// launch).
int enqueue_launch_profiled(lbm_t* h, int from, int steps, bool tail) {
  cudaEvent_t e[2];
  int rc = profiled_pair(h, 0, e);
  if (rc) return rc;
  cudaEventRecord(e[0], h->stream);
  enqueue_launch(h, from, steps, h->stream, false, tail);
  cudaEventRecord(e[1], h->stream);
  return LBM_OK;
}

}  // namespace

// Shared with the batched mode: the caller is capturing this stream into a
// graph of its own.
bool lbm_internal_capturing(cudaStream_t s) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (!s) return false;  // the legacy stream cannot be
  if (cudaStreamIsCapturing(s, &st) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return st == cudaStreamCaptureStatusActive;
}

namespace {

int check_launch() {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(LBM_ECUDA, "kernel launch failed: %s", cudaGetErrorString(e));
  return LBM_OK;
}

bool shape_compiled(int bx, int rows) {
  bool okb = false, okr = false;
  for (int v : kShapesBX) okb |= v == bx;
  for (int v : kShapesRows) okr |= v == rows;
  return okb && okr;
}

}  // namespace

// =========================================================================
// C ABI
// =========================================================================
extern "C" {

const char* lbm_last_error(void) { return g_last_error.c_str(); }

lbm_t* lbm_create(int32_t nx, int32_t ny, double tau, double farfield_rho, const double farfield_u[2]) {
  if (nx < 3 || ny < 3 || nx > 65536 || ny > 65536) {
    fail(LBM_EINVAL, "lbm_create: nx=%d ny=%d outside [3, 65536]", nx, ny);
    return nullptr;
  }
  if (!std::isfinite(tau) || !(tau > 0.5)) {
    fail(LBM_EINVAL, "lbm_create: tau=%g must be finite and > 0.5", tau);
    return nullptr;
  }
  if (!farfield_u || !std::isfinite(farfield_rho) || !(farfield_rho > 0.0) || !std::isfinite(farfield_u[0]) ||
      !std::isfinite(farfield_u[1])) {
    fail(LBM_EINVAL, "lbm_create: far field must be finite with rho > 0 and u non-NULL");
    return nullptr;
  }
  lbm_t* h = new lbm_t();
  h->nx = nx;
  h->ny = ny;
  h->tau = tau;
  h->nsbc.set(0.6, 0.0, 3.0, 0, 1);
  h->nsbc.m0[0] = farfield_rho;
  h->nsbc.m0[1] = farfield_u[0];
  h->nsbc.m0[2] = farfield_u[1];
  lbm_set_precision(h, LBM_F32);
  return h;
}

void lbm_destroy(lbm_t* h) {
  if (!h) return;
  if (h->stream || h->cap || h->bound) cudaStreamSynchronize(h->stream);
  if (h->moved) cudaDeviceSynchronize();  // steps on an earlier stream may still use the handle's slot
  drop_graphs(h);
  if (h->bound) {
    lbmk::check_remove(h->buf[0]);
    lbmk::check_remove(h->buf[1]);
  }
  if (h->owns_memory) {
    cudaFree(h->buf[0]);
    cudaFree(h->buf[1]);
    cudaFree(h->scratch);
  }
  for (cudaEvent_t e : h->ev_pool) cudaEventDestroy(e);
  give_sync(h);
  if (h->d_items) cudaFree(h->d_items);
  if (h->d_inst) cudaFree(h->d_inst);
  if (h->d_shift) cudaFree(h->d_shift);
  if (h->cap) {
    cudaStreamDestroy(h->cap);
    cudaStreamDestroy(h->side);
    cudaEventDestroy(h->ev_fork);
    cudaEventDestroy(h->ev_join);
    for (cudaEvent_t e : h->ev_chunk) cudaEventDestroy(e);
  }
  delete h;
}

int lbm_set_nsbc(lbm_t* h, double gamma, double beta, double kappa, int32_t corner_mode, int32_t grad_order) {
  if (!h) return fail(LBM_EINVAL, "lbm_set_nsbc: NULL handle");
  if (!std::isfinite(gamma) || !std::isfinite(beta) || !std::isfinite(kappa) || (grad_order != 1 && grad_order != 2) ||
      (corner_mode != LBM_CORNER_DIAGONAL && corner_mode != LBM_CORNER_MEAN))
    return fail(LBM_EINVAL, "lbm_set_nsbc: need finite gamma, beta, kappa, corner_mode 0 or 1 and grad_order 1 or 2");
  h->nsbc.set(gamma, beta, kappa, corner_mode, grad_order);
  drop_graphs(h);
  return LBM_OK;
}

}  // extern "C"

// Autotuner cache (lbm_set_tune_cache), shared with the batched mode: the
// file path ("" = off; the LBM_TUNE_CACHE environment variable sets it until
// the first lbm_set_tune_cache) and the hit / miss counts.
#ifndef LBM_BUILD_ID
#define LBM_BUILD_ID "unversioned"
#endif
namespace {
std::mutex g_tune_mutex;
std::string g_tune_path;
bool g_tune_set = false;
long long g_tune_hits = 0, g_tune_misses = 0;
}  // namespace

std::string lbm_internal_tune_path() {
  std::lock_guard<std::mutex> lock(g_tune_mutex);
  if (!g_tune_set) {
    const char* env = std::getenv("LBM_TUNE_CACHE");
    g_tune_path = env ? env : "";
    g_tune_set = true;
  }
  return g_tune_path;
}

// The key of a tuning problem on the current device (see lbm_tune_cache.h).
std::string lbm_internal_tune_key(const char* kind, int storage, int model, bool shift,
                                  const std::vector<long long>& dims) {
  int dev = 0, drv = 0, rt = 0;
  cudaGetDevice(&dev);
  cudaDriverGetVersion(&drv);
  cudaRuntimeGetVersion(&rt);
  cudaDeviceProp prop{};
  const char* name = cudaGetDeviceProperties(&prop, dev) == cudaSuccess ? prop.name : "unknown-device";
  return lbmtune::make_key(name, drv, rt, LBM_BUILD_ID, kind, storage, model, shift, dims);
}

void lbm_internal_tune_count(bool hit) {
  std::lock_guard<std::mutex> lock(g_tune_mutex);
  (hit ? g_tune_hits : g_tune_misses) += 1;
}

extern "C" int lbm_set_tune_cache(const char* path) {
  std::lock_guard<std::mutex> lock(g_tune_mutex);
  g_tune_path = path ? path : "";
  g_tune_set = true;
  return LBM_OK;
}

extern "C" int lbm_tune_cache_stats(int64_t* hits, int64_t* misses) {
  if (!hits || !misses) return fail(LBM_EINVAL, "lbm_tune_cache_stats: NULL argument");
  std::lock_guard<std::mutex> lock(g_tune_mutex);
  *hits = g_tune_hits;
  *misses = g_tune_misses;
  return LBM_OK;
}

// Shared with the batched mode: validate edge types and fill the NSBC block.
int lbm_internal_set_edges(lbmk::Nsbc* p, const int32_t types[4], const double uw[8]) {
  if (!types) return fail(LBM_EINVAL, "set_edges: NULL types");
  for (int s = 0; s < 4; ++s)
    if (types[s] < LBM_EDGE_NSBC || types[s] > LBM_EDGE_VELOCITY)
      return fail(LBM_EINVAL, "set_edges: unknown edge type %d on side %d", types[s], s);
  if ((types[0] == LBM_EDGE_PERIODIC) != (types[1] == LBM_EDGE_PERIODIC) ||
      (types[2] == LBM_EDGE_PERIODIC) != (types[3] == LBM_EDGE_PERIODIC))
    return fail(LBM_EINVAL, "set_edges: periodic edges come in pairs (left+right, bottom+top)");
  for (int s = 0; s < 4; ++s)
    if (types[s] == LBM_EDGE_VELOCITY && (!uw || !std::isfinite(uw[2 * s]) || !std::isfinite(uw[2 * s + 1])))
      return fail(LBM_EINVAL, "set_edges: velocity edge %d needs a finite velocity", s);
  p->periodic_x = types[0] == LBM_EDGE_PERIODIC;
  p->periodic_y = types[2] == LBM_EDGE_PERIODIC;
  for (int s = 0; s < 4; ++s) {
    p->vel[s] = types[s] == LBM_EDGE_VELOCITY;
    p->uw[s][0] = p->vel[s] ? uw[2 * s] : 0.0;
    p->uw[s][1] = p->vel[s] ? uw[2 * s + 1] : 0.0;
  }
  return LBM_OK;
}

extern "C" {

int lbm_set_edges(lbm_t* h, const int32_t types[4], const double uw[8]) {
  if (!h) return fail(LBM_EINVAL, "lbm_set_edges: NULL handle");
  lbmk::Nsbc p = h->nsbc;
  int rc = lbm_internal_set_edges(&p, types, uw);
  if (rc) return rc;
  h->nsbc = p;
  drop_graphs(h);
  return LBM_OK;
}

int lbm_set_collision(lbm_t* h, int32_t model, double omega_e, double omega_eps, double omega_q) {
  if (!h) return fail(LBM_EINVAL, "lbm_set_collision: NULL handle");
  if (model != LBM_BGK && model != LBM_MRT) return fail(LBM_EINVAL, "lbm_set_collision: unknown model %d", model);
  if (model == LBM_MRT)
    for (double r : {omega_e, omega_eps, omega_q})
      if (!std::isfinite(r) || !(r > 0.0) || !(r < 2.0))
        return fail(LBM_EINVAL, "lbm_set_collision: MRT rates must lie in (0, 2)");
  h->collision = model;
  if (model == LBM_MRT) {
    h->s_e = omega_e;
    h->s_eps = omega_eps;
    h->s_q = omega_q;
  }
  drop_graphs(h);
  return LBM_OK;
}

int lbm_set_precision(lbm_t* h, int32_t storage) {
  if (!h) return fail(LBM_EINVAL, "lbm_set_precision: NULL handle");
  if (storage < LBM_F64 || storage > LBM_BF16) return fail(LBM_EINVAL, "lbm_set_precision: unknown storage %d", storage);
  if (h->bound) return fail(LBM_ESTATE, "lbm_set_precision: memory already bound or allocated");
  h->storage = storage;
  h->elt = storage == LBM_F64 ? 8 : (storage == LBM_F32 ? 4 : 2);
  h->pitch = (int)round_up((size_t)h->nx, 64);
  h->plane = (long long)(round_up((size_t)h->ny * h->pitch * h->elt, 256) / h->elt);
  return LBM_OK;
}

int lbm_set_stream(lbm_t* h, void* cuda_stream) {
  if (!h) return fail(LBM_EINVAL, "lbm_set_stream: NULL handle");
  h->moved |= h->initialised && h->stream != static_cast<cudaStream_t>(cuda_stream);
  h->stream = static_cast<cudaStream_t>(cuda_stream);
  return LBM_OK;
}

size_t lbm_buffer_bytes(const lbm_t* h) { return h ? (size_t)9 * h->plane * h->elt : 0; }

size_t lbm_scratch_bytes(const lbm_t* h) {
  return h ? 3 * macro_bytes(h) + round_up((kReduceBlocks * 4 + 5) * sizeof(double), 256) : 0;
}

int lbm_bind(lbm_t* h, void* dev_a, void* dev_b, void* dev_scratch) {
  if (!h || !dev_a || !dev_b || !dev_scratch) return fail(LBM_EINVAL, "lbm_bind: NULL argument");
  if (h->bound) return fail(LBM_ESTATE, "lbm_bind: memory already bound or allocated");
  for (void* p : {dev_a, dev_b, dev_scratch})
    if (reinterpret_cast<uintptr_t>(p) % 256) return fail(LBM_EINVAL, "lbm_bind: pointers must be 256-byte aligned");
  LBM_CUDA(cudaGetDevice(&h->device));
  if (int rc = take_sync(h)) return rc;
  h->buf[0] = dev_a;
  h->buf[1] = dev_b;
  h->scratch = dev_scratch;
  lbmk::check_add(dev_a, lbm_buffer_bytes(h));  // bounds-checked build only
  lbmk::check_add(dev_b, lbm_buffer_bytes(h));
  h->bound = true;
  h->owns_memory = false;
  return LBM_OK;
}

int lbm_init_device(lbm_t* h, const double* d_rho, const double* d_ux, const double* d_uy) {
  if (!h || !d_rho || !d_ux || !d_uy) return fail(LBM_EINVAL, "lbm_init_device: NULL argument");
  int rc = ensure_memory(h);
  if (rc) return rc;
  h->cur = 0;
  h->waited = false;
  enqueue_init_rows(h, d_rho, d_ux, d_uy, 0, h->ny);
  rc = check_launch();
  if (rc) return rc;
  h->initialised = true;
  h->steps = 0;
  return LBM_OK;
}

int lbm_init(lbm_t* h, const double* rho, const double* ux, const double* uy) {
  LBM_TRACE("lbm_init");
  if (!h || !rho || !ux || !uy) return fail(LBM_EINVAL, "lbm_init: NULL argument");
  int rc = ensure_memory(h);
  if (rc) return rc;
  rc = ensure_streams(h);
  if (rc) return rc;
  h->waited = false;
  // the copy of row chunk c (side stream, copy engine) overlaps the
  // initialisation of chunk c - 1 (the handle's stream)
  const double* src[3] = {rho, ux, uy};
  LBM_CUDA(cudaEventRecord(h->ev_fork, h->stream));  // earlier work on the scratch area first
  LBM_CUDA(cudaStreamWaitEvent(h->side, h->ev_fork, 0));
  h->cur = 0;
  constexpr int K = (int)(sizeof(h->ev_chunk) / sizeof(h->ev_chunk[0]));
  for (int c = 0; c < K; ++c) {
    const int y0 = (int)((long long)h->ny * c / K), y1 = (int)((long long)h->ny * (c + 1) / K);
    if (y1 <= y0) continue;
    const size_t off = (size_t)y0 * h->nx, bytes = (size_t)(y1 - y0) * h->nx * sizeof(double);
    for (int f = 0; f < 3; ++f)
      LBM_CUDA(cudaMemcpyAsync(scratch_field(h, f) + off, src[f] + off, bytes, cudaMemcpyHostToDevice, h->side));
    LBM_CUDA(cudaEventRecord(h->ev_chunk[c], h->side));
    LBM_CUDA(cudaStreamWaitEvent(h->stream, h->ev_chunk[c], 0));
    enqueue_init_rows(h, scratch_field(h, 0), scratch_field(h, 1), scratch_field(h, 2), y0, y1);
  }
  rc = check_launch();
  if (rc) return rc;
  h->initialised = true;
  h->steps = 0;
  LBM_CUDA(cudaStreamSynchronize(h->stream));
  return LBM_OK;
}

int lbm_step(lbm_t* h, int32_t n) {
  LBM_TRACE("lbm_step");
  if (!h) return fail(LBM_EINVAL, "lbm_step: NULL handle");
  if (n < 0) return fail(LBM_EINVAL, "lbm_step: n=%d < 0", n);
  if (!h->initialised) return fail(LBM_ESTATE, "lbm_step: call lbm_init first");
  int rc = ensure_streams(h);
  if (!rc) rc = prepare_form(h);
  if (!rc && n >= kResidentMin) rc = prepare_resident(h);
  if (!rc) rc = ensure_staged(h);
  if (rc) return rc;
  const int per = steps_per_launch(h);
  // A caller's graph is replayed on the buffers it was captured with, so an
  // even number of steps must leave the state in the buffer it came from, as
  // single steps do: as many launches as that takes (and none of the graphs
  // below, which a capture does not take).
  const bool captured = lbm_internal_capturing(h->stream);
  long long launches = ((long long)n + per - 1) / per;
  launches += (launches ^ n) & 1;
  if (n > 0 && (h->form == Form::Pass || h->form == Form::Staged)) h->waited = true;
  int left = n;
  while (!captured && h->rs_halo && left >= kResidentMin) {
    const int take = std::min(left, kResidentMax);
    cudaEvent_t e[2];
    if (h->profiling) {
      rc = profiled_pair(h, 0, e);
      if (rc) return rc;
      cudaEventRecord(e[0], h->stream);
    }
    rc = enqueue_resident(h, take);
    if (rc) return rc;
    if (h->profiling) cudaEventRecord(e[1], h->stream);
    if (h->rs_halo)
      left -= take;
    else if (h->profiling)
      h->ev_used -= 2;  // refused: nothing was launched between the two
  }
  if (!captured && !h->profiling && per == 1 && left >= kGraphSteps) {
    if (!h->graph[h->cur]) {
      rc = capture_graph(h, h->cur);
      if (rc) return rc;
    }
    while (left >= kGraphSteps) {
      LBM_CUDA(cudaGraphLaunch(h->graph[h->cur], h->stream));
      left -= kGraphSteps;  // kGraphSteps is even: h->cur is unchanged
    }
  }
  int tail = !captured && left % kGraphSteps >= kTailSteps && tail_serves(h) ? left % kGraphSteps : 0;
  if (tail) {
    rc = prepare_tail(h);
    if (rc) return rc;
    if (h->tl_steps < 2) tail = 0;
  }
  while (left > 0) {
    const bool tiles = h->form == Form::Tiles || left <= tail;
    const int most = tiles ? h->tl_steps : per;
    int take = std::min(most, left);
    // a pass takes at least two steps: five are three and two, not four and one
    if (h->form == Form::Pass && left - take == 1 && take > 2) --take;
    // the last tile launches share what is left evenly
    if (tiles) take = (left + (left + most - 1) / most - 1) / ((left + most - 1) / most);
    if (captured) take = (int)((left + launches - 1) / launches--);
    if (!h->profiling)
      enqueue_launch(h, h->cur, take, h->stream, false, tiles);
    else
      rc = take > 1 || tiles ? enqueue_launch_profiled(h, h->cur, take, tiles) : enqueue_step_profiled(h, h->cur);
    if (rc) return rc;
    h->cur ^= 1;
    left -= take;
  }
  rc = check_launch();
  if (rc) return rc;
  h->steps += n;
  return LBM_OK;
}

int64_t lbm_steps_done(const lbm_t* h) { return h ? h->steps : -1; }

int lbm_get_dims(const lbm_t* h, int32_t* nx, int32_t* ny) {
  if (!h || !nx || !ny) return fail(LBM_EINVAL, "lbm_get_dims: NULL argument");
  *nx = h->nx;
  *ny = h->ny;
  return LBM_OK;
}

namespace lbmk {
void batch_check_read(unsigned long long* count, unsigned long long* first, bool reset);  // lbm_batch.cu
}

int lbm_check_read(int64_t* rejected, uint64_t* first_address, int32_t reset) {
  if (!rejected || !first_address) return fail(LBM_EINVAL, "lbm_check_read: NULL argument");
  unsigned long long c1 = 0, f1 = 0, c2 = 0, f2 = 0;
  lbmk::check_read(&c1, &f1, reset != 0);
  lbmk::batch_check_read(&c2, &f2, reset != 0);
  *rejected = (int64_t)(c1 + c2);
  *first_address = c1 ? f1 : f2;
  return lbmk::kChecked ? 1 : 0;
}

int lbm_get_macros_device(lbm_t* h, double* d_rho, double* d_ux, double* d_uy) {
  if (!h || !d_rho || !d_ux || !d_uy) return fail(LBM_EINVAL, "lbm_get_macros_device: NULL argument");
  if (!h->initialised) return fail(LBM_ESTATE, "lbm_get_macros_device: call lbm_init first");
  enqueue_macros_rows(h, d_rho, d_ux, d_uy, 0, h->ny);
  return check_launch();
}

int lbm_get_macros(lbm_t* h, double* rho, double* ux, double* uy) {
  LBM_TRACE("lbm_get_macros");
  if (!h || !rho || !ux || !uy) return fail(LBM_EINVAL, "lbm_get_macros: NULL argument");
  if (!h->initialised) return fail(LBM_ESTATE, "lbm_get_macros: call lbm_init first");
  int rc = ensure_streams(h);
  if (rc) return rc;
  // the macros of row chunk c (the handle's stream) overlap the copy-out of
  // chunk c - 1 (side stream, copy engine)
  double* dst[3] = {rho, ux, uy};
  constexpr int K = (int)(sizeof(h->ev_chunk) / sizeof(h->ev_chunk[0]));
  for (int c = 0; c < K; ++c) {
    const int y0 = (int)((long long)h->ny * c / K), y1 = (int)((long long)h->ny * (c + 1) / K);
    if (y1 <= y0) continue;
    enqueue_macros_rows(h, scratch_field(h, 0), scratch_field(h, 1), scratch_field(h, 2), y0, y1);
    LBM_CUDA(cudaEventRecord(h->ev_chunk[c], h->stream));
    LBM_CUDA(cudaStreamWaitEvent(h->side, h->ev_chunk[c], 0));
    const size_t off = (size_t)y0 * h->nx, bytes = (size_t)(y1 - y0) * h->nx * sizeof(double);
    for (int f = 0; f < 3; ++f)
      LBM_CUDA(cudaMemcpyAsync(dst[f] + off, scratch_field(h, f) + off, bytes, cudaMemcpyDeviceToHost, h->side));
  }
  rc = check_launch();
  if (rc) return rc;
  LBM_CUDA(cudaEventRecord(h->ev_join, h->side));  // later work on the handle's stream waits for the copies
  LBM_CUDA(cudaStreamWaitEvent(h->stream, h->ev_join, 0));
  return sync_checked(h, h->side, "lbm_get_macros");
}

int lbm_get_populations(lbm_t* h, double* f) {
  if (!h || !f) return fail(LBM_EINVAL, "lbm_get_populations: NULL argument");
  if (!h->initialised) return fail(LBM_ESTATE, "lbm_get_populations: call lbm_init first");
  const long long n = (long long)h->nx * h->ny;
  for (int i = 0; i < 9; ++i) {
    dispatch(h->storage, [&](auto tag) {
      using T = decltype(tag);
      lbmk::plane_to_f64<T><<<grid_for(n, 256), 256, 0, h->stream>>>(static_cast<const T*>(h->buf[h->cur]), geom(h),
                                                                      zshift(h), i, scratch_field(h, 0));
    });
    int rc = check_launch();
    if (rc) return rc;
    LBM_CUDA(cudaMemcpyAsync(f + i * n, scratch_field(h, 0), n * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    LBM_CUDA(cudaStreamSynchronize(h->stream));
  }
  return sync_checked(h, h->stream, "lbm_get_populations");
}

int lbm_set_populations(lbm_t* h, const double* f) {
  if (!h || !f) return fail(LBM_EINVAL, "lbm_set_populations: NULL argument");
  int rc = ensure_memory(h);
  if (!rc) rc = clear_sched(h);
  if (rc) return rc;
  const long long n = (long long)h->nx * h->ny;
  h->cur = 0;
  for (int i = 0; i < 9; ++i) {
    LBM_CUDA(cudaMemcpyAsync(scratch_field(h, 0), f + i * n, n * sizeof(double), cudaMemcpyHostToDevice, h->stream));
    dispatch(h->storage, [&](auto tag) {
      using T = decltype(tag);
      for (int b = 0; b < 2; ++b)
        lbmk::f64_to_plane<T><<<grid_for((long long)h->ny * h->pitch, 256), 256, 0, h->stream>>>(
            static_cast<T*>(h->buf[b]), geom(h), zshift(h), i, scratch_field(h, 0));
    });
    rc = check_launch();
    if (rc) return rc;
    LBM_CUDA(cudaStreamSynchronize(h->stream));
  }
  h->initialised = true;
  h->steps = 0;
  return LBM_OK;
}

}  // extern "C"

// Checkpoint record: this header, then the population buffer as stored.
namespace {
struct StateHeader {
  char magic[8];  // "LBMSTAT1"
  int32_t version, storage, nx, ny, pitch, reserved;
  int64_t steps;
  double m0[3];  // far field: the stored populations are deviations from f^eq(m0)
};
static_assert(sizeof(StateHeader) == 64, "checkpoint header layout");
constexpr char kStateMagic[8] = {'L', 'B', 'M', 'S', 'T', 'A', 'T', '1'};
}  // namespace

extern "C" {

size_t lbm_state_bytes(const lbm_t* h) { return h ? sizeof(StateHeader) + lbm_buffer_bytes(h) : 0; }

int lbm_save_state(lbm_t* h, void* host, size_t bytes, int64_t* steps) {
  if (!h || !host) return fail(LBM_EINVAL, "lbm_save_state: NULL argument");
  if (!h->initialised) return fail(LBM_ESTATE, "lbm_save_state: call lbm_init first");
  if (bytes != lbm_state_bytes(h))
    return fail(LBM_EINVAL, "lbm_save_state: %zu bytes given, the record is %zu", bytes, lbm_state_bytes(h));
  StateHeader hd{};
  std::memcpy(hd.magic, kStateMagic, sizeof hd.magic);
  hd.version = 1;
  hd.storage = h->storage;
  hd.nx = h->nx;
  hd.ny = h->ny;
  hd.pitch = h->pitch;
  hd.steps = h->steps;
  for (int c = 0; c < 3; ++c) hd.m0[c] = h->nsbc.m0[c];
  std::memcpy(host, &hd, sizeof hd);
  LBM_CUDA(cudaMemcpyAsync(static_cast<char*>(host) + sizeof hd, h->buf[h->cur], lbm_buffer_bytes(h),
                           cudaMemcpyDeviceToHost, h->stream));
  if (steps) *steps = h->steps;
  return sync_checked(h, h->stream, "lbm_save_state");
}

int lbm_load_state(lbm_t* h, const void* host, size_t bytes) {
  if (!h || !host) return fail(LBM_EINVAL, "lbm_load_state: NULL argument");
  if (bytes != lbm_state_bytes(h))
    return fail(LBM_EINVAL, "lbm_load_state: %zu bytes given, the record is %zu", bytes, lbm_state_bytes(h));
  // the record must describe this handle's layout and far field, or its
  // bytes mean something else here
  StateHeader hd;
  std::memcpy(&hd, host, sizeof hd);
  if (std::memcmp(hd.magic, kStateMagic, sizeof hd.magic) != 0 || hd.version != 1)
    return fail(LBM_EINVAL, "lbm_load_state: not a checkpoint record of this library");
  if (hd.storage != h->storage || hd.nx != h->nx || hd.ny != h->ny || hd.pitch != h->pitch)
    return fail(LBM_EINVAL, "lbm_load_state: record holds storage %d, %d x %d (pitch %d); handle has %d, %d x %d (%d)",
                hd.storage, hd.nx, hd.ny, hd.pitch, h->storage, h->nx, h->ny, h->pitch);
  for (int c = 0; c < 3; ++c)
    if (std::memcmp(&hd.m0[c], &h->nsbc.m0[c], sizeof(double)) != 0)
      return fail(LBM_EINVAL, "lbm_load_state: record's far field (%.17g, %.17g, %.17g) differs from the handle's",
                  hd.m0[0], hd.m0[1], hd.m0[2]);
  if (hd.steps < 0) return fail(LBM_EINVAL, "lbm_load_state: step count %lld < 0", (long long)hd.steps);
  int rc = ensure_memory(h);
  if (!rc) rc = clear_sched(h);
  if (rc) return rc;
  h->cur = 0;
  const size_t bb = lbm_buffer_bytes(h);
  LBM_CUDA(cudaMemcpyAsync(h->buf[0], static_cast<const char*>(host) + sizeof hd, bb, cudaMemcpyHostToDevice,
                           h->stream));
  LBM_CUDA(cudaMemcpyAsync(h->buf[1], h->buf[0], bb, cudaMemcpyDeviceToDevice, h->stream));
  LBM_CUDA(cudaStreamSynchronize(h->stream));
  h->initialised = true;
  h->steps = hd.steps;
  return LBM_OK;
}

int lbm_reduce(lbm_t* h, const double* ref_rho, const double* ref_ux, const double* ref_uy, int32_t ref_pitch,
               double out[4]) {
  LBM_TRACE("lbm_reduce");
  if (!h || !out) return fail(LBM_EINVAL, "lbm_reduce: NULL argument");
  if (!h->initialised) return fail(LBM_ESTATE, "lbm_reduce: call lbm_init first");
  if (ref_rho && (!ref_ux || !ref_uy || ref_pitch < h->nx))
    return fail(LBM_EINVAL, "lbm_reduce: reference needs rho, ux, uy and pitch >= nx");
  lbmk::RefField ref{ref_rho, ref_ux, ref_uy, ref_pitch};
  const long long n = (long long)h->nx * h->ny;
  const int blocks = (int)std::min<long long>(kReduceBlocks, (n + kReduceThreads - 1) / kReduceThreads);
  dispatch(h->storage, [&](auto tag) {
    using T = decltype(tag);
    lbmk::reduce_kernel<T, kReduceThreads><<<blocks, kReduceThreads, 0, h->stream>>>(
        static_cast<const T*>(h->buf[h->cur]), geom(h), lbmk::shift_as<typename lbmk::Store<T>::C>(zshift(h)), ref,
        h->nsbc.m0[0], h->nsbc.m0[1], h->nsbc.m0[2], scratch_partials(h));
  });
  lbmk::reduce_finish<kReduceThreads><<<1, kReduceThreads, 0, h->stream>>>(scratch_partials(h), blocks, scratch_out(h),
                                                                         sched(h) + 2);
  int rc = check_launch();
  if (rc) return rc;
  double sums[5];
  LBM_CUDA(cudaMemcpyAsync(sums, scratch_out(h), sizeof sums, cudaMemcpyDeviceToHost, h->stream));
  LBM_CUDA(cudaStreamSynchronize(h->stream));
  std::memcpy(out, sums, 4 * sizeof(double));
  if (sums[4] != 0.0) return fail(LBM_ETIMEOUT, "lbm_reduce: a bounded wait of a step kernel gave up");
  if (out[3] > 0.0) return fail(LBM_EUNSTABLE, "lbm_reduce: %.0f nodes with non-finite or non-positive density", out[3]);
  return LBM_OK;
}

int lbm_profile(lbm_t* h, int32_t enable) {
  if (!h) return fail(LBM_EINVAL, "lbm_profile: NULL handle");
  h->profiling = enable != 0;
  h->ev_used = 0;
  return LBM_OK;
}

int lbm_profile_read(lbm_t* h, double out[4]) {
  if (!h || !out) return fail(LBM_EINVAL, "lbm_profile_read: NULL argument");
  LBM_CUDA(cudaStreamSynchronize(h->stream));
  double ms[2] = {0.0, 0.0}, n[2] = {0.0, 0.0};
  for (size_t k = 0; k + 1 < h->ev_used; k += 2) {
    float t = 0.f;
    LBM_CUDA(cudaEventElapsedTime(&t, h->ev_pool[k], h->ev_pool[k + 1]));
    ms[h->ev_kind[k]] += t;
    n[h->ev_kind[k]] += 1.0;
  }
  out[0] = ms[0];
  out[1] = n[0];
  out[2] = ms[1];
  out[3] = n[1];
  h->ev_used = 0;
  return LBM_OK;
}

int lbm_set_launch(lbm_t* h, int32_t threads_x, int32_t rows, int32_t prefetch_rows) {
  if (!h) return fail(LBM_EINVAL, "lbm_set_launch: NULL handle");
  if (threads_x == 0 && rows == 0) {
    threads_x = 128;
    rows = 1;
  }
  if (!shape_compiled(threads_x, rows))
    return fail(LBM_EINVAL, "lbm_set_launch: shape (%d, %d) not compiled", threads_x, rows);
  if (prefetch_rows < 0 || prefetch_rows > 64)
    return fail(LBM_EINVAL, "lbm_set_launch: prefetch_rows=%d outside [0, 64]", prefetch_rows);
  h->bx = threads_x;
  h->rows = rows;
  h->pf = prefetch_rows;
  h->staged = 0;
  h->fused = false;
  h->twostep = false;
  h->tiles = false;
  h->form_auto = false;
  drop_graphs(h);
  return LBM_OK;
}

int lbm_set_fused(lbm_t* h, int32_t enable) {
  if (!h) return fail(LBM_EINVAL, "lbm_set_fused: NULL handle");
  h->fused = enable != 0;
  h->form_auto = false;
  if (h->fused) {
    h->staged = 0;
    h->twostep = false;
    h->tiles = false;
  }
  drop_graphs(h);
  return LBM_OK;
}

int32_t lbm_get_fused(const lbm_t* h) { return h ? (h->fused ? 1 : 0) : LBM_EINVAL; }

int lbm_set_staged(lbm_t* h, int32_t stages) {
  if (!h) return fail(LBM_EINVAL, "lbm_set_staged: NULL handle");
  if (stages != 0 && stages != 3 && stages != 4)
    return fail(LBM_EINVAL, "lbm_set_staged: stages=%d (0 = off, 3 or 4)", stages);
  h->staged = stages;
  h->form_auto = false;
  if (stages) {
    h->fused = false;
    h->twostep = false;
    h->tiles = false;
  }
  drop_graphs(h);
  return LBM_OK;
}

int32_t lbm_get_staged(const lbm_t* h) { return h ? h->staged : LBM_EINVAL; }

int lbm_set_twostep(lbm_t* h, int32_t enable) {
  if (!h) return fail(LBM_EINVAL, "lbm_set_twostep: NULL handle");
  if (enable && !pass_ok(h))
    return fail(LBM_EINVAL, "lbm_set_twostep: needs f32, f16 or bf16 storage, no periodic axis and 8 x 8 nodes or more");
  h->twostep = enable != 0;
  h->form_auto = false;
  if (h->twostep) {
    h->staged = 0;
    h->fused = false;
    h->tiles = false;
  }
  drop_graphs(h);
  return LBM_OK;
}

int lbm_set_tiles(lbm_t* h, int32_t enable) {
  if (!h) return fail(LBM_EINVAL, "lbm_set_tiles: NULL handle");
  if (enable) {
    int rc = device_sms(h);
    if (rc) return rc;
    if (!tiles_ok(h) || (long long)h->nx * h->ny > kTileCells || tile_plan(h).steps == 0)
      return fail(LBM_EINVAL, "lbm_set_tiles: needs 8 x 8 to %lld nodes that tiles in shared memory can cover", kTileCells);
  }
  h->tiles = enable != 0;
  h->form_auto = false;
  if (h->tiles) {
    h->staged = 0;
    h->fused = false;
    h->twostep = false;
  }
  drop_graphs(h);
  return LBM_OK;
}

int lbm_get_form(lbm_t* h, int32_t* form, int32_t* steps_per_launch, int32_t* resident_from) {
  if (!h || !form || !steps_per_launch || !resident_from) return fail(LBM_EINVAL, "lbm_get_form: NULL argument");
  if (!h->bound) return fail(LBM_ESTATE, "lbm_get_form: no memory yet (lbm_bind or lbm_init first)");
  int rc = prepare_form(h);
  if (!rc) rc = prepare_resident(h);
  if (rc) return rc;
  *form = (int32_t)h->form;
  *steps_per_launch = ::steps_per_launch(h);
  *resident_from = h->rs_halo ? kResidentMin : 0;
  return LBM_OK;
}

int32_t lbm_get_twostep(const lbm_t* h) { return h ? (h->twostep ? 1 : 0) : LBM_EINVAL; }

int lbm_status(lbm_t* h) {
  if (!h) return fail(LBM_EINVAL, "lbm_status: NULL handle");
  if (!h->initialised) return LBM_OK;  // nothing has run
  return sync_checked(h, h->stream, "lbm_status");
}

int lbm_set_wait_limit(lbm_t* h, int64_t cycles) {
  if (!h) return fail(LBM_EINVAL, "lbm_set_wait_limit: NULL handle");
  if (cycles < 0 || cycles > 4000000000LL)
    return fail(LBM_EINVAL, "lbm_set_wait_limit: %lld outside [0, 4e9] cycles", (long long)cycles);
  h->wait_limit = (unsigned)cycles;
  return LBM_OK;
}

int lbm_autotune(lbm_t* h, int32_t* threads_x, int32_t* rows, int32_t* prefetch_rows, double* ms_per_step) {
  LBM_TRACE("lbm_autotune");
  if (!h) return fail(LBM_EINVAL, "lbm_autotune: NULL handle");
  if (!h->initialised) return fail(LBM_ESTATE, "lbm_autotune: call lbm_init first");
  int rc = ensure_streams(h);
  if (rc) return rc;
  // a choice recorded for the same key is applied without timing
  const std::string tune_path = lbm_internal_tune_path();
  std::string tune_key;
  if (!tune_path.empty()) {
    tune_key = lbm_internal_tune_key("domain", h->storage, h->collision, zshift(h).on, {h->nx, h->ny});
    lbmtune::Entry e;
    double bx = 0, r = 0, pf = 0, st = -1, fz = -1, ts = -1, tl = -1, ms = 0;
    if (lbmtune::lookup(tune_path, tune_key, &e) && e.get("threads_x", &bx) && e.get("rows", &r) &&
        e.get("prefetch_rows", &pf) && e.get("staged", &st) && e.get("fused", &fz) && e.get("twostep", &ts) &&
        e.get("tiles", &tl) && e.get("ms_per_step", &ms) && (st == 0 || st == 3 || st == 4) && (fz == 0 || fz == 1) &&
        (ts == 0 || ts == 1) && (tl == 0 || (tl == 1 && tiles_ok(h))) && lbm_set_launch(h, (int32_t)bx, (int32_t)r, (int32_t)pf) == LBM_OK &&
        (st == 0 || lbm_set_staged(h, (int32_t)st) == LBM_OK) && (fz == 0 || lbm_set_fused(h, 1) == LBM_OK) &&
        (ts == 0 || lbm_set_twostep(h, 1) == LBM_OK)) {
      h->tiles = tl == 1;
      lbm_internal_tune_count(true);
      if (threads_x) *threads_x = h->bx;
      if (rows) *rows = h->rows;
      if (prefetch_rows) *prefetch_rows = h->pf;
      if (ms_per_step) *ms_per_step = ms;
      return LBM_OK;
    }
  }
  // keep the state: copy the current buffer aside, restore it at the end
  const size_t bb = lbm_buffer_bytes(h);
  void* backup = nullptr;
  LBM_CUDA(cudaMallocAsync(&backup, bb, h->stream));
  LBM_CUDA(cudaMemcpyAsync(backup, h->buf[h->cur], bb, cudaMemcpyDeviceToDevice, h->stream));
  cudaEvent_t e0, e1;
  LBM_CUDA(cudaEventCreate(&e0));
  LBM_CUDA(cudaEventCreate(&e1));
  const long long cells = (long long)h->nx * h->ny;
  const int reps = (int)std::max<long long>(4, std::min<long long>(64, (1LL << 28) / std::max(cells, 1LL)));
  float best = 1e30f;
  int best_bx = h->bx, best_rows = h->rows, best_pf = h->pf, best_staged = h->staged;
  bool best_fused = h->fused, best_twostep = false, best_tiles = false;
  h->twostep = h->tiles = h->form_auto = false;
  // whole steps as the graphs run them (NSBC kernel on the forked branch)
  auto time_steps = [&]() -> float {
    h->form_ready = false;
    if (prepare_form(h) != LBM_OK) return 1e30f;
    for (int k = 0; k < 2; ++k) enqueue_step(h, k & 1, h->stream, true);
    cudaEventRecord(e0, h->stream);
    for (int k = 0; k < reps; ++k) enqueue_step(h, k & 1, h->stream, true);
    cudaEventRecord(e1, h->stream);
    if (cudaEventSynchronize(e1) != cudaSuccess) return 1e30f;
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    return ms / reps;
  };
  // small domains: steps as lbm_step replays them (captured graphs of
  // kGraphSteps steps), since there the gaps between launches are part of
  // what is being chosen (timed one by one, a form with fewer launches per
  // step looks better than it runs)
  const bool use_graph = cells <= (1LL << 22);
  auto time_graph = [&]() -> float {
    drop_graphs(h);
    if (prepare_form(h) != LBM_OK || ensure_staged(h) != LBM_OK) return 1e30f;
    if (capture_graph(h, 0) != LBM_OK) return 1e30f;
    const int n = std::max(1, reps / kGraphSteps);
    cudaGraphLaunch(h->graph[0], h->stream);
    cudaEventRecord(e0, h->stream);
    for (int k = 0; k < n; ++k) cudaGraphLaunch(h->graph[0], h->stream);
    cudaEventRecord(e1, h->stream);
    float ms = 1e30f;
    if (cudaEventSynchronize(e1) == cudaSuccess) {
      cudaEventElapsedTime(&ms, e0, e1);
      ms /= (float)(n * kGraphSteps);
    }
    drop_graphs(h);
    return ms;
  };
  auto time_form = [&]() -> float { return use_graph ? time_graph() : time_steps(); };
  h->staged = 0;
  for (int bx : kShapesBX)
    for (int r : kShapesRows)
      for (int pf : kPrefetchRows)
        for (bool fz : {false, true}) {  // the kernel pair, or both in one launch
          if (r > 1 && (h->ny - 2) / r < 152) continue;  // too few blocks to fill the GPU
          h->bx = bx;
          h->rows = r;
          h->pf = pf;
          h->fused = fz;
          const float ms = time_form();
          if (ms < best) {
            best = ms;
            best_bx = bx;
            best_rows = r;
            best_pf = pf;
            best_staged = 0;
            best_fused = fz;
            best_twostep = false;
          }
        }
  h->fused = false;
  // the staged step kernel (producer/consumer, 3 or 4 tile stages)
  for (int st : {3, 4}) {
    h->staged = st;
    drop_graphs(h);
    if (ensure_staged(h) != LBM_OK) break;
    const float ms = time_form();
    if (ms < best) {
      best = ms;
      best_staged = st;
      best_fused = false;
      best_twostep = false;
    }
  }
  // the forms of several steps per launch, launched as lbm_step does
  h->staged = 0;
  for (bool tiles : {false, true}) {
    if (tiles ? !tiles_ok(h) || cells > kTileCells : !pass_ok(h)) continue;
    h->twostep = !tiles;
    h->tiles = tiles;
    drop_graphs(h);
    if (prepare_form(h) == LBM_OK && prepare_resident(h) == LBM_OK &&
        h->form == (tiles ? Form::Tiles : Form::Pass)) {
      const int cur = h->cur;
      if (h->rs_halo) enqueue_resident(h, kResidentMin);  // (moves h->cur; finds out whether it is launched at all)
      const bool resident = h->rs_halo != 0;
      const int per = resident ? kResidentMin : steps_per_launch(h), launches = resident ? 2 : std::max(4, reps / per);
      auto launch = [&](int k) {
        if (resident)
          enqueue_resident(h, per);
        else
          enqueue_launch(h, k & 1, per, h->stream, false, false);
      };
      for (int k = 0; k < (resident ? 1 : 2); ++k) launch(k);
      cudaEventRecord(e0, h->stream);
      for (int k = 0; k < launches; ++k) launch(k);
      cudaEventRecord(e1, h->stream);
      h->cur = cur;
      float ms = 1e30f;
      if (cudaEventSynchronize(e1) == cudaSuccess) {
        cudaEventElapsedTime(&ms, e0, e1);
        ms /= (float)(per * launches);
      }
      if (ms < best) {
        best = ms;
        best_twostep = !tiles;
        best_tiles = tiles;
        best_staged = 0;
        best_fused = false;
      }
    }
    h->twostep = h->tiles = false;
  }
  rc = check_launch();
  h->bx = best_bx;
  h->rows = best_rows;
  h->pf = best_pf;
  h->staged = best_staged;
  h->fused = best_fused && !best_staged;
  h->twostep = best_twostep;
  h->tiles = best_tiles;
  drop_graphs(h);
  LBM_CUDA(cudaMemcpyAsync(h->buf[h->cur], backup, bb, cudaMemcpyDeviceToDevice, h->stream));
  LBM_CUDA(cudaFreeAsync(backup, h->stream));
  LBM_CUDA(cudaStreamSynchronize(h->stream));
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc) return rc;
  if (!tune_path.empty()) {
    lbm_internal_tune_count(false);
    lbmtune::Entry e{tune_key,
                     {{"threads_x", best_bx}, {"rows", best_rows}, {"prefetch_rows", best_pf},
                      {"staged", h->staged}, {"fused", h->fused ? 1 : 0}, {"twostep", h->twostep ? 1 : 0},
                      {"tiles", h->tiles ? 1 : 0}, {"ms_per_step", best}}};
    lbmtune::store(tune_path, e);  // a cache that cannot be written is only not reused
  }
  if (threads_x) *threads_x = best_bx;
  if (rows) *rows = best_rows;
  if (prefetch_rows) *prefetch_rows = best_pf;
  if (ms_per_step) *ms_per_step = best;
  return LBM_OK;
}

}  // extern "C"

// =========================================================================
// Allocation-free reduction (lbm_reduce_noalloc).
//
// Some callers cannot allocate device memory at the moment they want the
// reduction: a monitoring hook that runs inside another framework's step
// loop, where that framework owns the device memory (its caching allocator
// holds it) or where cudaMalloc/cudaFree would synchronise the device and
// stall the framework's other streams.  For them, lbm_reduce_noalloc runs the
// same reduction kernels as lbm_reduce but keeps the per-block partial sums
// and the four results in the fixed array below instead of the handle's
// scratch area.  It calls no cudaMalloc, cudaFree or allocating routine.
//
// The array lives in every GPU that loads this library until the process
// exits.  Every call on a device shares it and it keeps the last call's
// contents; nothing in it needs to start at zero, because a call reads only
// slots that the same call wrote first.  Calls that overlap on the GPU
// (other streams, other host threads, other handles on the same device) race
// on it: the caller must order them.
// =========================================================================
namespace {

// reduce_kernel hands whole rows to blocks (row y to block y mod grid) and
// columns to threads, so any domain works with at most kNoAllocMaxBlocks
// blocks: the grid is min(ny, kNoAllocMaxBlocks), one block per row up to that.
constexpr int kNoAllocThreads = kReduceThreads;
constexpr int kNoAllocMaxBlocks = 4096;
constexpr int kNoAllocDoubles = kNoAllocMaxBlocks * 4 + 5;  // partials + out[5]: 131,112 bytes

static __device__ __align__(256) double g_noalloc_scratch[kNoAllocDoubles];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mutex;
double* g_noalloc_ptr[kMaxDevices] = {};

// Device address of g_noalloc_scratch on the current device.  In host code
// the array's name is only a host-side stand-in, so the address is looked up
// once per device (with that device current) and cached.
int noalloc_scratch(double** out) {
  int dev = 0;
  LBM_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return fail(LBM_EINVAL, "lbm_reduce_noalloc: device %d out of range", dev);
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p)
      return fail(LBM_ECUDA, "lbm_reduce_noalloc: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
    g_noalloc_ptr[dev] = static_cast<double*>(p);
  }
  *out = g_noalloc_ptr[dev];
  return LBM_OK;
}

}  // namespace

extern "C" int lbm_reduce_noalloc(lbm_t* h, const double* ref_rho, const double* ref_ux, const double* ref_uy,
                                  int32_t ref_pitch, double out[4]) {
  if (!h || !out) return fail(LBM_EINVAL, "lbm_reduce_noalloc: NULL argument");
  const int blocks = std::min(h->ny, kNoAllocMaxBlocks);
  if (!h->initialised) return fail(LBM_ESTATE, "lbm_reduce_noalloc: call lbm_init first");
  if (ref_rho && (!ref_ux || !ref_uy || ref_pitch < h->nx))
    return fail(LBM_EINVAL, "lbm_reduce_noalloc: reference needs rho, ux, uy and pitch >= nx");
  if (h->bound) {
    int dev = -1;
    LBM_CUDA(cudaGetDevice(&dev));
    if (dev != h->device) return fail(LBM_EINVAL, "lbm_reduce_noalloc: handle lives on device %d, current is %d",
                                      h->device, dev);
  }
  double* scratch = nullptr;
  int rc = noalloc_scratch(&scratch);
  if (rc) return rc;
  double* partials = scratch;
  double* d_out = scratch + kNoAllocMaxBlocks * 4;
  lbmk::RefField ref{ref_rho, ref_ux, ref_uy, ref_pitch};
  dispatch(h->storage, [&](auto tag) {
    using T = decltype(tag);
    lbmk::reduce_kernel<T, kNoAllocThreads><<<blocks, kNoAllocThreads, 0, h->stream>>>(
        static_cast<const T*>(h->buf[h->cur]), geom(h), lbmk::shift_as<typename lbmk::Store<T>::C>(zshift(h)), ref,
        h->nsbc.m0[0], h->nsbc.m0[1], h->nsbc.m0[2], partials);
  });
  lbmk::reduce_finish<kNoAllocThreads><<<1, kNoAllocThreads, 0, h->stream>>>(partials, blocks, d_out, sched(h) + 2);
  rc = check_launch();
  if (rc) return rc;
  double sums[5];
  LBM_CUDA(cudaMemcpyAsync(sums, d_out, sizeof sums, cudaMemcpyDeviceToHost, h->stream));
  LBM_CUDA(cudaStreamSynchronize(h->stream));
  std::memcpy(out, sums, 4 * sizeof(double));
  if (sums[4] != 0.0) return fail(LBM_ETIMEOUT, "lbm_reduce_noalloc: a bounded wait of a step kernel gave up");
  if (out[3] > 0.0)
    return fail(LBM_EUNSTABLE, "lbm_reduce_noalloc: %.0f nodes with non-finite or non-positive density", out[3]);
  return LBM_OK;
}
