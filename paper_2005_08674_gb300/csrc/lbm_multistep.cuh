// lbm_multistep.cuh -- several time steps per pass over a domain (temporal
// blocking): the state is read from device memory once and written once for
// kPassSteps steps, with the bits of as many single steps.  Two ways of
// keeping the steps in between on chip:
//
//   rolling items (roll_item): a warp owns a strip of 64 columns and rolls
//       down a band of rows.  It stages the state rows by bulk copies in a
//       private ring in shared memory and carries, for each step in between,
//       the populations that the next step pulls in registers, rounded to
//       the storage type as a single step stores them.  Every node it needs
//       is an interior node at every step, so it holds no boundary code: it
//       serves the nodes at distance kPassSteps or more from every edge.
//   tiles (tile_steps): a block stages a rectangle and a halo as wide as the
//       number of steps in shared memory and advances it there, boundary
//       nodes (Sec. 5) included.  The nodes near the edges of a large domain
//       (its frame) are such tiles, and a small domain is nothing but tiles.
//
// Neither waits for another block: what an item needs it computes itself.
#pragma once

#include "lbm_kernels.cuh"
#include "lbm_staged.cuh"

namespace lbmk {

constexpr int kPassSteps = 4;  // most steps per pass of the rolling kernels (2 .. 4)

// ---------------------------------------------------------------------------
// Tiles.
// ---------------------------------------------------------------------------
// Output nodes [x0, x1) x [y0, y1) of a tile.
struct TileRect {
  int x0, y0, x1, y1;
};

// A step's state of a tile in shared memory, in stored units as the compute
// type: population i of local node (lx, ly) at (9 ly + i) w + lx.  ld / st
// take domain coordinates and physical units like GlobalSrc / GlobalDst; on
// a periodic axis a coordinate may lie a period away from the tile's.
template <typename T>
struct TileState {
  using C = typename Store<T>::C;
  C* s;
  int rx0, ry0, w, nx, ny;
  __device__ __forceinline__ int at(int i, int x, int y, int lw, int lh) const {
    int lx = x - rx0, ly = y - ry0;
    lx = lx < 0 ? lx + nx : (lx >= lw ? lx - nx : lx);
    ly = ly < 0 ? ly + ny : (ly >= lh ? ly - ny : ly);
    return (9 * ly + i) * w + lx;
  }
  int h;
  __device__ __forceinline__ C ld(int i, int x, int y) const {
    const C v = s[at(i, x, y, w, h)];
    if constexpr (Store<T>::kScale == 1)
      return v;
    else
      return v * C(1.0 / Store<T>::kScale);
  }
  __device__ __forceinline__ void st(int i, int x, int y, C v) const {
    const T t = Store<T>::cvt(v);
    s[at(i, x, y, w, h)] = Store<T>::ld1s(&t);
  }
};

// v rounded to the storage type, as a step stores it (stored units).
template <typename T>
__device__ __forceinline__ typename Store<T>::C stored(typename Store<T>::C v) {
  if constexpr (sizeof(T) == sizeof(typename Store<T>::C)) {
    return v;
  } else {
    const T t = T(v);
    return Store<T>::ld1s(&t);
  }
}

// 4 and 8 bytes from global to shared memory without a register.
template <typename T>
__device__ __forceinline__ void tile_copy(T* dst, const T* src) {
  if (!in_bounds(src, sizeof(T))) {
    *dst = 0;
    return;
  }
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(dst)), "l"(src), "n"(sizeof(T)) : "memory");
}

// Shared memory of a tile of region w x h: two steps' states.
template <typename C>
__host__ __device__ constexpr size_t tile_bytes(int w, int h) {
  return (size_t)2 * 9 * w * h * sizeof(C);
}

// `steps` steps of the output nodes `t` (A: step n, B: step n + steps), by a
// block of NT threads.  Step j is computed on the output rectangle widened by
// steps - j nodes on each side (clipped at the domain's edges, running past
// them along a periodic axis), so the last one needs no other tile's results.
// Sides of the rectangle that lie on an edge are at least two nodes deep:
// the second-order difference reads the node two further in.
template <typename T, int MODEL, bool SHIFT, int NT>
__device__ __forceinline__ void tile_steps(const T* __restrict__ A, T* __restrict__ B, const Geom& g, const Nsbc& p,
                                           const Rates<typename Store<T>::C>& r, const TileRect& t, int steps,
                                           typename Store<T>::C* smem) {
  using S = Store<T>;
  using C = typename S::C;
  const int tid = threadIdx.x;
  const bool px = p.periodic_x != 0, py = p.periodic_y != 0;
  const int rx0 = px ? t.x0 - steps : max(t.x0 - steps, 0), rx1 = px ? t.x1 + steps : min(t.x1 + steps, g.nx);
  const int ry0 = py ? t.y0 - steps : max(t.y0 - steps, 0), ry1 = py ? t.y1 + steps : min(t.y1 + steps, g.ny);
  const int w = rx1 - rx0, h = ry1 - ry0;
  const int other = 9 * w * h;  // the two steps' states: smem and smem + other
  // element e of the region's state: population k % 9 of row k / 9, k = e / w
  // (the factor is exact: e w < 2^32).  Asynchronous copies, or eight loads
  // of 16-bit values at once, keep every load of the tile in flight.
  const unsigned mul_w = 0xffffffffu / (unsigned)w + 1u;
  auto source = [&](int e) {
    const int k = (int)__umulhi(mul_w, (unsigned)e), lx = e - k * w;
    const int ly = k / 9, i = k - 9 * ly;
    int x = rx0 + lx, y = ry0 + ly;
    x = x < 0 ? x + g.nx : (x >= g.nx ? x - g.nx : x);
    y = y < 0 ? y + g.ny : (y >= g.ny ? y - g.ny : y);
    return A + i * g.plane + (long long)y * g.pitch + x;
  };
  if constexpr (sizeof(T) >= 4) {
#pragma unroll 4
    for (int e = tid; e < other; e += NT) tile_copy<T>(smem + e, source(e));
  } else {
    for (int e0 = tid; e0 < other; e0 += 8 * NT) {
      C v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = e0 + q * NT < other ? S::ld1(source(e0 + q * NT)) : C(0);
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (e0 + q * NT < other) smem[e0 + q * NT] = v[q];
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  for (int j = 1; j <= steps; ++j) {
    const C* __restrict__ src = smem + (j & 1 ? 0 : other);
    C* __restrict__ dst = smem + (j & 1 ? other : 0);
    const bool last = j == steps;
    const int e = steps - j;
    const int ax = px ? t.x0 - e : max(t.x0 - e, 0), bx = px ? t.x1 + e : min(t.x1 + e, g.nx);
    const int ay = py ? t.y0 - e : max(t.y0 - e, 0), by = py ? t.y1 + e : min(t.y1 + e, g.ny);
    // perimeter rows and columns inside the step's rectangle (along a
    // periodic axis also their images a period away)
    const int wj = bx - ax, hj = by - ay;
    int n_rows = 0, n_cols = 0, rows[4], cols[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int yk = k == 0 ? 0 : (k == 1 ? g.ny - 1 : (k == 2 ? -1 : g.ny));
      const int xk = k == 0 ? 0 : (k == 1 ? g.nx - 1 : (k == 2 ? -1 : g.nx));
      rows[k] = yk;
      cols[k] = xk;
      const bool ry = (k < 2 || py) && yk >= ay && yk < by, rx = (k < 2 || px) && xk >= ax && xk < bx;
      n_rows |= ry << k;  // bit k: row rows[k] lies inside
      n_cols |= rx << k;
    }
    const int n_per = __popc(n_rows) * wj + __popc(n_cols) * hj;
    const int edge_slots = (4 * n_per + 31) & ~31;
    // interior nodes: the rectangle without the edges of non-periodic axes
    const int ix = px ? ax : max(ax, 1), jx = px ? bx : min(bx, g.nx - 1);
    const int iy = py ? ay : max(ay, 1), jy = py ? by : min(by, g.ny - 1);
    const int wi = max(jx - ix, 0), n_int = wi * max(jy - iy, 0);
    constexpr bool PAIR = std::is_same<C, float>::value;
    const int n_work = PAIR ? (n_int + 1) >> 1 : n_int;
    // q / wi = high word of q mul: exact, n_int * wi < 2^32; a width of 1 has no such factor
    const unsigned mul = wi > 1 ? 0xffffffffu / (unsigned)wi + 1u : 0u;  // ceil(2^32 / wi)
    for (int u = tid; u < edge_slots + n_work; u += NT) {
      if (u < edge_slots) {
        // a boundary node per quad of lanes
        int k = u >> 2;
        if (k >= n_per) continue;
        int x = 0, y = 0;
        bool found = false, twice = false;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (!found && (n_rows >> c & 1)) {
            if (k < wj) {
              found = true;
              x = ax + k;
              y = rows[c];
            } else {
              k -= wj;
            }
          }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (!found && (n_cols >> c & 1)) {
            if (k < hj) {
              found = true;
              x = cols[c];
              y = ay + k;
#pragma unroll
              for (int d = 0; d < 4; ++d) twice |= (n_rows >> d & 1) && rows[d] == y;  // already taken with its row
            } else {
              k -= hj;
            }
          }
        }
        if (!found || twice) continue;
        EdgeNode en[1];
        const bool ok[1] = {true};
        en[0].x = x < 0 ? x + g.nx : (x >= g.nx ? x - g.nx : x);
        en[0].y = y < 0 ? y + g.ny : (y >= g.ny ? y - g.ny : y);
        en[0].nxn = px ? 0 : (en[0].x == 0 ? -1 : (en[0].x == g.nx - 1 ? 1 : 0));
        en[0].nyn = py ? 0 : (en[0].y == 0 ? -1 : (en[0].y == g.ny - 1 ? 1 : 0));
        en[0].open = en[0].nxn != 0 || en[0].nyn != 0;
        const TileState<T> from{const_cast<C*>(src), rx0, ry0, w, g.nx, g.ny, h};
        if (last)
          nsbc_edge_nodes<T, MODEL, 1, SHIFT>(from, GlobalDst<T>{B, g.plane, g.pitch}, g, p, r, en, ok, tid & 3);
        else
          nsbc_edge_nodes<T, MODEL, 1, SHIFT>(from, TileState<T>{dst, rx0, ry0, w, g.nx, g.ny, h}, g, p, r, en, ok,
                                              tid & 3);
        continue;
      }
      constexpr int N = PAIR ? 2 : 1;  // two nodes at once in float (paired FP32 instructions)
      C v[9][N];
      int at[N], gx[N], gy[N];
      bool ok[N];
#pragma unroll
      for (int k = 0; k < N; ++k) {
        const int q = u - edge_slots + k * n_work;
        ok[k] = q < n_int;
        const int qq = ok[k] ? q : 0;
        const int row = wi > 1 ? (int)__umulhi(mul, (unsigned)qq) : qq;
        gy[k] = iy + row;
        gx[k] = ix + (qq - row * wi);
        if (px) ok[k] = ok[k] && gx[k] != 0 && gx[k] != g.nx - 1 && gx[k] != -1 && gx[k] != g.nx;
        if (py) ok[k] = ok[k] && gy[k] != 0 && gy[k] != g.ny - 1 && gy[k] != -1 && gy[k] != g.ny;
        at[k] = 9 * (gy[k] - ry0) * w + (gx[k] - rx0);
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i][k] = src[at[k] + (i - 9 * cy(i)) * w - cx(i)];
      }
      collide_nodes<MODEL, SHIFT, PAIR>(v, r, C(S::kScale));
#pragma unroll
      for (int k = 0; k < N; ++k) {
        if (!ok[k]) continue;
        if (last) {
          const int x = gx[k] < 0 ? gx[k] + g.nx : (gx[k] >= g.nx ? gx[k] - g.nx : gx[k]);
          const int y = gy[k] < 0 ? gy[k] + g.ny : (gy[k] >= g.ny ? gy[k] - g.ny : gy[k]);
          T* o = B + (long long)y * g.pitch + x;
#pragma unroll
          for (int i = 0; i < 9; ++i) S::st1r(o + i * g.plane, v[i][k]);
        } else {
#pragma unroll
          for (int i = 0; i < 9; ++i) dst[at[k] + i * w] = stored<T>(v[i][k]);
        }
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// The frame of a domain (nodes closer than D, the pass's steps, to an edge) as
// tiles of the rolling kernels' blocks: the first and last D rows in pieces
// along x, then the first and last D columns of the rows between along y.
// ---------------------------------------------------------------------------
constexpr int kFrameLength = 40;  // longest piece: its region fits a block's shared memory

__host__ __device__ inline int frame_pieces(int n) { return n <= 0 ? 0 : (n + kFrameLength - 1) / kFrameLength; }
// their number (the same for every D; the shortest pass has two steps)
__host__ __device__ inline int frame_tiles(int nx, int ny) { return 2 * frame_pieces(nx) + 2 * frame_pieces(ny - 4); }
// tile k of them; empty (y0 = y1) where no rows are left between
__host__ __device__ inline TileRect frame_tile(int nx, int ny, int D, int k) {
  const int nh = frame_pieces(nx);
  TileRect t;
  if (k < 2 * nh) {
    const int q = k >> 1;
    t.x0 = (int)((unsigned)nx * q / nh);
    t.x1 = (int)((unsigned)nx * (q + 1) / nh);
    t.y0 = k & 1 ? ny - D : 0;
    t.y1 = t.y0 + D;
  } else {
    k -= 2 * nh;
    const int m = ny - 2 * D, nv = frame_pieces(ny - 4), q = k >> 1;
    t.y0 = D + (int)((unsigned)m * q / nv);
    t.y1 = D + (int)((unsigned)m * (q + 1) / nv);
    t.x0 = k & 1 ? nx - D : 0;
    t.x1 = t.x0 + D;
  }
  return t;
}

// ---------------------------------------------------------------------------
// The rolling interior.
// ---------------------------------------------------------------------------
template <typename T>
struct Roll {
  static constexpr int K = kPassSteps;
  static constexpr int W = 64;  // state columns of a strip, two per lane
  // output columns of a strip: step n + j is valid on columns j .. W - 1 - j,
  // and strips start OUT apart, a multiple of 16 bytes for the copies
  static constexpr int OUT = (W - 2 * K) / (16 / (int)sizeof(T)) * (16 / (int)sizeof(T));
  static constexpr int DEPTH = 6;  // ring rows: three read, the others in flight
  // resident blocks per SM.  The kernel waits on its own chain of operations
  // (57 % of issue slots used with three blocks), so what counts is how many
  // warps the registers allow.  f32 carries 54 registers: three blocks (168).
  // 16 bits carried as stored pairs are 27: four (128), 8192^2 f16 259 -> 247
  // us a step, 3001 x 1777 bf16 29.7 -> 27.1; a fifth (96) spills and gives
  // 245 and 27.3, but 273 against 262 in a mean flow.
  static constexpr int BLOCKS = sizeof(T) == 4 ? 3 : 4;
  static constexpr int ROWE = 9 * W;
  static constexpr int WARPS = 4;  // independent warps per block
  static constexpr size_t kRing = (size_t)WARPS * DEPTH * ROWE * sizeof(T);
  static constexpr size_t kTile = tile_bytes<float>(kFrameLength + 2 * K, 2 * K);
  static constexpr size_t kSmem = kRing > kTile ? kRing : kTile;
};
constexpr int kRollThreads = 32 * 4;
constexpr bool kPinConst = true;

// this lane's two values of one population at columns 2 lane, 2 lane + 1 of
// a staged row, in stored units
__device__ __forceinline__ float2 roll_lds(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ float2 roll_lds(const __half* p) {
  return __half22float2(*reinterpret_cast<const __half2*>(p));
}
__device__ __forceinline__ float2 roll_lds(const __nv_bfloat16* p) {
  return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p));
}
// What an item carries of two neighbouring nodes' values of one population
// from row to row: the values rounded to the storage type, as a single step
// stores them, 16-bit ones as the pair they are stored as.
template <typename T>
struct RollPair;
template <>
struct RollPair<float> {
  float2 v;
  static __device__ __forceinline__ RollPair of(float2 a) { return {a}; }
  __device__ __forceinline__ float2 get() const { return v; }
};
template <>
struct RollPair<__half> {
  __half2 v;
  static __device__ __forceinline__ RollPair of(float2 a) { return {__floats2half2_rn(a.x, a.y)}; }
  __device__ __forceinline__ float2 get() const { return __half22float2(v); }
};
template <>
struct RollPair<__nv_bfloat16> {
  __nv_bfloat162 v;
  static __device__ __forceinline__ RollPair of(float2 a) { return {__floats2bfloat162_rn(a.x, a.y)}; }
  __device__ __forceinline__ float2 get() const { return __bfloat1622float2(v); }
};
// two neighbouring nodes' values of one population to device memory
__device__ __forceinline__ void roll_st(float* p, float2 v) {
  if (in_bounds(p, 8)) __stcs(reinterpret_cast<float2*>(p), v);
}
__device__ __forceinline__ void roll_st(__half* p, float2 v) {
  if (!in_bounds(p, 4)) return;
  const __half2 h = __floats2half2_rn(v.x, v.y);
  unsigned u;
  memcpy(&u, &h, 4);
  __stcs(reinterpret_cast<unsigned*>(p), u);
}
__device__ __forceinline__ void roll_st(__nv_bfloat16* p, float2 v) {
  if (!in_bounds(p, 4)) return;
  const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
  unsigned u;
  memcpy(&u, &h, 4);
  __stcs(reinterpret_cast<unsigned*>(p), u);
}

// v := the values at columns 2 lane - c, 2 lane + 1 - c (c = c_ix), i.e. what
// the lane's nodes pull along x; the strip's outermost columns get values
// that no valid node uses
__device__ __forceinline__ void shift_x(int c, float2& v) {
  if (c > 0) {
    const float l = __shfl_up_sync(0xffffffffu, v.y, 1);
    v.y = v.x;
    v.x = l;
  } else if (c < 0) {
    const float l = __shfl_down_sync(0xffffffffu, v.x, 1);
    v.x = v.y;
    v.y = l;
  }
}

template <typename T>
__device__ __forceinline__ void shift_x(int c, RollPair<T>& p) {
  if constexpr (sizeof(T) == 4) {
    shift_x(c, p.v);
  } else {
    unsigned v;
    memcpy(&v, &p.v, 4);
    if (c > 0)
      v = __byte_perm(__shfl_up_sync(0xffffffffu, v, 1), v, 0x5432);  // {left's second, first}
    else if (c < 0)
      v = __byte_perm(v, __shfl_down_sync(0xffffffffu, v, 1), 0x5432);  // {second, right's first}
    memcpy(&p.v, &v, 4);
  }
}

// The rows of a strip on their way into the ring: lanes 0..8 copy one
// population each (columns X0 .. X0 + W, clipped to the pitch).
// (Checked build: a copy whose range fails is neither issued nor counted.)
template <typename T>
struct RollStage {
  const T* src;    // this lane's population in the next row
  uint32_t bytes;  // per population and row
  uint32_t bar0;   // shared address of the ring's first barrier
  uint32_t dst0;   // and of this lane's population in the ring's first row
  int pitch, lane;
  // copies the next row into ring row `slot`
  __device__ __forceinline__ void row(int slot) {
    using R = Roll<T>;
    const bool ok = lane < 9 && in_bounds(src, bytes) &&
                    in_slot((long long)lane * R::W * (long long)sizeof(T), bytes, (long long)R::ROWE * sizeof(T));
    const uint32_t total = kChecked ? __reduce_add_sync(0xffffffffu, ok ? bytes : 0u) : 9 * bytes;
    const uint32_t bar = bar0 + 8 * slot;
    if (lane == 0)
      asm volatile("{ .reg .b64 st; mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1; }" ::"r"(bar), "r"(total)
                   : "memory");
    __syncwarp();
    if (ok)
      asm volatile(
          "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
              dst0 + slot * (uint32_t)(R::ROWE * sizeof(T))),
          "l"(src), "r"(bytes), "r"(bar)
          : "memory");
    src += pitch;
  }
};

// What a rolling item carries from row to row for step n + j, j = 1 .. K - 1,
// all already pulled along x: of the newest row r the c_y = 0 (mid) and c_y =
// +1 (up1) populations, and of row r - 1 the c_y = +1 ones (up2).
template <typename T>
struct RollCarry {
  RollPair<T> up2[kPassSteps - 1][3], mid[kPassSteps - 1][3], up1[kPassSteps - 1][3];
};

// State row s (ring slot `slot`) has arrived: step n + j of row s - j for j =
// 1 .. K, each from the row before it and what was carried of the two above,
// and the store of step n + K.  FULL: the rows above exist at every step
// (and K = kPassSteps), so nothing is conditional and every value stays in
// the register it was computed in; otherwise only the steps that have their
// rows are formed (s0: the item's first state row).
template <bool FULL, typename T, int MODEL, bool SHIFT>
__device__ __forceinline__ void roll_row(RollStage<T>& stage, T*& out, const Geom& g,
                                         const Rates<typename Store<T>::C>& r, int K, int x0, int s0, int s, int s1,
                                         int slot, const T* ring, int lo, int hi, bool whole, bool some, RollCarry<T>& c,
                                         const CellConst<float2>& k) {
  using R = Roll<T>;
  using S = Store<T>;
  constexpr int KM = R::K;
  // step n + 1 of row s - 1 from state rows s - 2, s - 1, s
  const int slot_m1 = slot == 0 ? R::DEPTH - 1 : slot - 1;
  const int slot_m2 = slot_m1 == 0 ? R::DEPTH - 1 : slot_m1 - 1;
  float2 h[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const int row = cy(i) > 0 ? slot_m2 : (cy(i) == 0 ? slot_m1 : slot);
    h[i] = roll_lds(ring + row * R::ROWE + i * R::W);
    shift_x(cx(i), h[i]);
  }
  // row s - 2 is read: stage row s + DEPTH - 2 in its place
  __syncwarp();
  if (s + R::DEPTH - 2 <= s1) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    stage.row(slot_m2);
  }
  collide<MODEL, SHIFT>(h, r, float(S::kScale), k);
  bool live = true;
#pragma unroll
  for (int j = 1; j < KM; ++j) {
    if (FULL || (live && j < K)) {
      // h: step n + j of row s - j
      RollPair<T> n[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        n[i] = RollPair<T>::of(h[i]);
        shift_x(cx(i), n[i]);
      }
      float2 o[9];
      o[0] = c.mid[j - 1][0].get();
      o[1] = c.mid[j - 1][1].get();
      o[2] = c.mid[j - 1][2].get();
      o[3] = c.up2[j - 1][0].get();
      o[5] = c.up2[j - 1][1].get();
      o[7] = c.up2[j - 1][2].get();
      o[4] = n[4].get();
      o[6] = n[6].get();
      o[8] = n[8].get();
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        c.up2[j - 1][a] = c.up1[j - 1][a];
        c.up1[j - 1][a] = n[3 + 2 * a];
        c.mid[j - 1][a] = n[a];
      }
      if (!FULL) live = s >= s0 + 2 * (j + 1);  // the rows above exist from here on
      if (FULL || live) {
        collide<MODEL, SHIFT>(o, r, float(S::kScale), k);
#pragma unroll
        for (int i = 0; i < 9; ++i) h[i] = o[i];
      }
    }
  }
  if (FULL || live) {
    if (whole) {
#pragma unroll
      for (int i = 0; i < 9; ++i) roll_st(out + i * g.plane, h[i]);
    } else if (some) {
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        if (x0 >= lo && x0 < hi) S::st1r(out + i * g.plane, h[i].x);
        if (x0 + 1 >= lo && x0 + 1 < hi) S::st1r(out + i * g.plane + 1, h[i].y);
      }
    }
    out += g.pitch;
  }
}

// One work item: steps n + 1 .. n + K (K = `steps`, at most kPassSteps) of
// output rows [Ya, Yb) x columns X0 + K .. X0 + K + OUT (clipped to [K, nx -
// K)) of the domain g, rolling down state rows Ya - K .. Yb + K - 1 through
// this warp's ring (rows `ring`, barriers `bar`, their parities in `phase`).
// All lanes of the warp call it.  The rows that fill the carry are formed
// step by step; the others two at a time, so that what is carried changes
// its name and not its register (one row per turn moved 87 registers per
// step, more than the 55 operations of the collision).  false: a wait gave
// up (err[2] is set).
template <typename T, int MODEL, bool SHIFT>
__device__ __forceinline__ bool roll_item(const T* __restrict__ A, T* __restrict__ B, const Geom& g,
                                          const Rates<typename Store<T>::C>& r, int K, int X0, int Ya, int Yb,
                                          T* ring, uint64_t* bar, uint32_t& phase, int lane, int* __restrict__ err) {
  using R = Roll<T>;
  const int s0 = Ya - K, s1 = Yb + K - 1;  // state rows read: s0 .. s1
  __syncwarp();                            // the previous item's reads of the ring are done
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  RollStage<T> stage{A + (lane < 9 ? lane : 0) * g.plane + (long long)s0 * g.pitch + X0,
                     (uint32_t)(min(X0 + R::W, g.pitch) - X0) * (uint32_t)sizeof(T), smem_u32(bar),
                     smem_u32(ring) + lane * (uint32_t)(R::W * sizeof(T)), g.pitch, lane};
  for (int k = 0; k < min(R::DEPTH, s1 - s0 + 1); ++k) stage.row(k);
  RollCarry<T> c;
#pragma unroll
  for (int j = 0; j < R::K - 1; ++j)
#pragma unroll
    for (int a = 0; a < 3; ++a) c.up2[j][a] = c.mid[j][a] = c.up1[j][a] = RollPair<T>::of(make_float2(0.f, 0.f));
  const int x0 = X0 + 2 * lane;
  T* out = B + (long long)Ya * g.pitch + x0;  // the lane's nodes of the next row stored
  const int lo = X0 + K, hi = min(g.nx - K, X0 + K + R::OUT);
  const bool whole = x0 >= lo && x0 + 2 <= hi;
  const bool some = !whole && x0 + 2 > lo && x0 < hi;
  const CellConst<float2> k = cell_const<MODEL, kPinConst && !SHIFT, float2>(r, float(Store<T>::kScale));
  const T* mine = ring + 2 * lane;
  int slot = 0;
  auto wait = [&](int sl) {
    const bool done = mbar_wait(&bar[sl], (phase >> sl) & 1u);
    phase ^= 1u << sl;
    if (__all_sync(0xffffffffu, done)) return true;
    if (lane == 0) atomicExch(&err[2], 1);
    return false;
  };
  auto next = [](int sl) { return sl + 1 == R::DEPTH ? 0 : sl + 1; };
  int s = s0;
  for (;;) {
    if (K == R::K && s >= s0 + 2 * R::K) {
#pragma unroll 1
      for (; s < s1; s += 2) {
        if (!wait(slot)) return false;
        roll_row<true, T, MODEL, SHIFT>(stage, out, g, r, K, x0, s0, s, s1, slot, mine, lo, hi, whole, some, c, k);
        slot = next(slot);
        if (!wait(slot)) return false;
        roll_row<true, T, MODEL, SHIFT>(stage, out, g, r, K, x0, s0, s + 1, s1, slot, mine, lo, hi, whole, some, c, k);
        slot = next(slot);
      }
    }
    if (s > s1) break;
    if (!wait(slot)) return false;
    if (s >= s0 + 2)
      roll_row<false, T, MODEL, SHIFT>(stage, out, g, r, K, x0, s0, s, s1, slot, mine, lo, hi, whole, some, c, k);
    slot = next(slot);
    ++s;
  }
  return true;
}

// The whole pass in one launch, A (step n) -> B (step n + steps).  Each block
// first takes its share of the n_tiles frame tiles, then its four warps claim
// rolling items from a counter (sched[0]): item j = (strip, band) reads
// columns X0 = strip OUT .. X0 + W and stores rows steps + b band .. + band of
// band b; items come as all strips of a band side by side, the bands in waves
// (wave k: bands k, k + n_waves, ...), so that the lines neighbouring strips
// share and the rows a band restarts on are read from L2.  The last warp out
// resets the counters.  A wait that gives up sets sched[2].
template <typename T, int MODEL, bool SHIFT>
__global__ void __launch_bounds__(kRollThreads, Roll<T>::BLOCKS)
    pass_kernel(const T* __restrict__ A, T* __restrict__ B, Geom g, Nsbc p, Rates<typename Store<T>::C> r,
                int steps, int n_tiles, int n_strips, int band, int n_bands, int bands_per_wave, int n_waves,
                int* __restrict__ sched) {
  using R = Roll<T>;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bars[R::WARPS][R::DEPTH];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  T* ring = reinterpret_cast<T*>(smem_raw) + warp * R::DEPTH * R::ROWE;
  uint64_t* bar = bars[warp];
  if (lane == 0) {
#pragma unroll
    for (int j = 0; j < R::DEPTH; ++j) mbar_init(&bar[j], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  for (int k = blockIdx.x; k < n_tiles; k += gridDim.x) {
    const TileRect t = frame_tile(g.nx, g.ny, steps, k);
    if (t.y0 < t.y1)
      tile_steps<T, MODEL, SHIFT, kRollThreads>(A, B, g, p, r, t, steps, reinterpret_cast<float*>(smem_raw));
  }
  uint32_t phase = 0u;  // bit j: parity of the next completion of bar[j]
  const int per_wave = bands_per_wave * n_strips, n_items = n_waves * per_wave;
  for (;;) {
    int c = 0;
    if (lane == 0) c = atomicAdd(&sched[0], 1);
    c = __shfl_sync(0xffffffffu, c, 0);
    if (c >= n_items) break;
    const int wave = c / per_wave, rem = c - wave * per_wave;
    const int m = rem / n_strips, strip = rem - m * n_strips;
    const int b = m * n_waves + wave;
    if (b >= n_bands) continue;
    const int Ya = steps + b * band, Yb = min(Ya + band, g.ny - steps);
    if (Ya >= Yb) continue;
    if (!roll_item<T, MODEL, SHIFT>(A, B, g, r, steps, strip * R::OUT, Ya, Yb, ring, bar, phase, lane, sched)) return;
  }
  if (lane == 0) {
    __threadfence();
    if (atomicAdd(&sched[1], 1) == (int)gridDim.x * R::WARPS - 1) {
      sched[0] = 0;
      __threadfence();
      sched[1] = 0;
    }
  }
}

// ---------------------------------------------------------------------------
// A small domain as tiles: gx x gy of them, one block each.
// ---------------------------------------------------------------------------
constexpr int kTileThreads = 512;

template <typename T, int MODEL, bool SHIFT>
__global__ void __launch_bounds__(kTileThreads)
    tile_kernel(const T* __restrict__ A, T* __restrict__ B, Geom g, Nsbc p, Rates<typename Store<T>::C> r, int gx,
                int gy, int steps) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int ty = blockIdx.x / gx, tx = blockIdx.x - ty * gx;
  // 32-bit divisions: nx gx < 2^32
  const TileRect t{(int)((unsigned)g.nx * tx / gx), (int)((unsigned)g.ny * ty / gy),
                   (int)((unsigned)g.nx * (tx + 1) / gx), (int)((unsigned)g.ny * (ty + 1) / gy)};
  tile_steps<T, MODEL, SHIFT, kTileThreads>(A, B, g, p, r, t, steps,
                                            reinterpret_cast<typename Store<T>::C*>(smem_raw));
}

constexpr size_t kTileRoom = 227 * 1024;  // shared memory of a block

// Host: gx x gy tiles and `steps` steps per launch, by a model of a launch: one
// block per SM, so the tiles run in waves of the SM count; a block loads its
// region, then each step costs a fixed latency and so much per node of the
// step's rectangle (it shrinks by a node on each inner side per step) and
// per boundary node.
struct TilePlan {
  int gx = 0, gy = 0, steps = 0, smem = 0;
  double us = 1e30;  // per step
};

inline TilePlan plan_tiles(int nx, int ny, bool f64, bool px, bool py, int sms) {
  // microseconds, measured: launch, load per node, step, node, boundary node
  const double t_launch = 2.0, t_load = f64 ? 1.4e-3 : 0.7e-3, t_step = f64 ? 0.9 : 0.35;
  const double t_node = f64 ? 15e-3 : 0.45e-3, t_edge = f64 ? 100e-3 : 3e-3;
  const size_t elt = f64 ? 8 : 4, room = kTileRoom;
  TilePlan best;
  for (int steps : {1, 2, 3, 4, 5, 6, 8, 10, 12})
    for (int gx = 1; gx <= 64 && nx / gx >= 4; ++gx)
      for (int gy = 1; gy <= 64 && ny / gy >= 4; ++gy) {
        if (gx * gy > 8 * sms) break;
        const int tw = (nx + gx - 1) / gx, th = (ny + gy - 1) / gy;
        const int w = px || gx > 2 ? tw + 2 * steps : (gx == 2 ? tw + steps : tw);
        const int h = py || gy > 2 ? th + 2 * steps : (gy == 2 ? th + steps : th);
        if ((px && w > nx) || (py && h > ny)) continue;
        const size_t smem = 2 * 9 * (size_t)w * h * elt;
        if (smem > room) continue;
        const int waves = (gx * gy + sms - 1) / sms;
        double block = 0.8 + t_load * w * h;
        for (int j = 1; j <= steps; ++j) {
          const double c = (double)(steps - j) / steps;  // of the halo that step j still covers
          const double wj = tw + (w - tw) * c, hj = th + (h - th) * c;
          block += t_step + t_node * wj * hj + t_edge * std::max(wj, hj);
        }
        const double us = (t_launch + waves * block) / steps;
        if (us < best.us) best = TilePlan{gx, gy, steps, (int)smem, us};
      }
  return best;
}

// ---------------------------------------------------------------------------
// The same pass over many independent instances (the batched mode): the
// instance table, per-instance storage shifts and relaxation rates as the
// batched single step takes them, so the bits are those of batched steps.
// ---------------------------------------------------------------------------
template <typename C, bool SHIFT>
__device__ __forceinline__ Rates<C> instance_rates(const InstDev& d, const Shift<C>* __restrict__ shifts, int k,
                                                   double s_e, double s_eps, double s_q) {
  Rates<C> r{C(d.omega), C(s_e), C(s_eps), C(s_q), {}};
  if constexpr (SHIFT) r.z = shifts[k];
  return r;
}

// Frame tiles {instance k, tile, 0, 0}, shared out over the blocks; then
// rolling items {instance k, strip start X0, output rows Ya, Yb} (clipped to
// the rows at distance `steps` or more), claimed by warps from sched[0] (the
// last warp to finish resets it and sched[1]), largest instance first, all
// strips of a band side by side.
template <typename T, int MODEL, bool SHIFT>
__global__ void __launch_bounds__(kRollThreads, Roll<T>::BLOCKS)
    pass_batch_kernel(const T* __restrict__ A, T* __restrict__ B, const InstDev* __restrict__ inst,
                      const Shift<typename Store<T>::C>* __restrict__ shifts, const int4* __restrict__ tiles,
                      int n_tiles, const int4* __restrict__ items, int n_items, int steps, Nsbc p, double s_e,
                      double s_eps, double s_q, int* __restrict__ sched) {
  using R = Roll<T>;
  using C = typename Store<T>::C;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bars[R::WARPS][R::DEPTH];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  T* ring = reinterpret_cast<T*>(smem_raw) + warp * R::DEPTH * R::ROWE;
  uint64_t* bar = bars[warp];
  if (lane == 0) {
#pragma unroll
    for (int j = 0; j < R::DEPTH; ++j) mbar_init(&bar[j], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  for (int j = blockIdx.x; j < n_tiles; j += gridDim.x) {
    const int4 w = tiles[j];
    const InstDev d = inst[w.x];
    const Rates<C> r = instance_rates<C, SHIFT>(d, shifts, w.x, s_e, s_eps, s_q);
    Nsbc q = p;
    q.m0[0] = d.m0[0];
    q.m0[1] = d.m0[1];
    q.m0[2] = d.m0[2];
    const Geom g{d.nx, d.ny, d.pitch, d.plane};
    const TileRect t = frame_tile(d.nx, d.ny, steps, w.y);
    if (t.y0 < t.y1)
      tile_steps<T, MODEL, SHIFT, kRollThreads>(A + d.off, B + d.off, g, q, r, t, steps,
                                                reinterpret_cast<float*>(smem_raw));
  }
  uint32_t phase = 0u;
  for (;;) {
    int c = 0;
    if (lane == 0) c = atomicAdd(&sched[0], 1);
    c = __shfl_sync(0xffffffffu, c, 0);
    if (c >= n_items) break;
    const int4 w = items[c];
    const InstDev d = inst[w.x];
    const Rates<C> r = instance_rates<C, SHIFT>(d, shifts, w.x, s_e, s_eps, s_q);
    const Geom g{d.nx, d.ny, d.pitch, d.plane};
    const int Ya = max(w.z, steps), Yb = min(w.w, d.ny - steps);
    if (Ya >= Yb) continue;
    if (!roll_item<T, MODEL, SHIFT>(A + d.off, B + d.off, g, r, steps, w.y, Ya, Yb, ring, bar, phase, lane, sched))
      return;
  }
  if (lane == 0) {
    __threadfence();
    if (atomicAdd(&sched[1], 1) == (int)gridDim.x * R::WARPS - 1) {
      sched[0] = 0;
      sched[1] = 0;
    }
  }
}

}  // namespace lbmk
