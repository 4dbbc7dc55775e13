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
// Neither waits for another block: what an item needs it computes itself.  A
// domain whose state fits the SMs' shared memory can also stay there for all
// the steps of a call (resident_kernel); its blocks exchange halos.
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

// The region of a tile: its output nodes and `halo` more on each side, cut at
// the domain's edges and running past them along a periodic axis.
struct TileRegion {
  int x0, y0, w, h;
};

__host__ __device__ inline TileRegion tile_region(int nx, int ny, bool px, bool py, const TileRect& t, int halo) {
  const int x0 = px || t.x0 > halo ? t.x0 - halo : 0, x1 = px || t.x1 + halo < nx ? t.x1 + halo : nx;
  const int y0 = py || t.y0 > halo ? t.y0 - halo : 0, y1 = py || t.y1 + halo < ny ? t.y1 + halo : ny;
  return TileRegion{x0, y0, x1 - x0, y1 - y0};
}

// The state of the region, from A to shared memory, by a block of NT threads.
template <typename T, int NT>
__device__ __forceinline__ void tile_load(const T* __restrict__ A, const Geom& g, const TileRegion& reg,
                                          typename Store<T>::C* smem) {
  using S = Store<T>;
  using C = typename S::C;
  const int tid = threadIdx.x, w = reg.w, rx0 = reg.x0, ry0 = reg.y0;
  const int other = 9 * w * reg.h;
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
}

// ---- boundary nodes of a resident tile --------------------------------------
// Where a quad of lanes finds its boundary node, worked out once per launch:
// nsbc_edge_nodes, which serves any source, looks its node up and wraps every
// address anew in each step, half of the instructions of a chain that all
// the other warps of the block wait for.
struct EdgeSlot {
  int x, y;      // may lie past the domain along a periodic axis
  int at, back;  // the node's population 0 in the region's state; the same of this lane's node b - q n
  EdgeNode en;   // the node's own coordinates and normal
  bool any, kp, km, want;  // a node; its pulled pair is known; the lane's node b - q n is needed
};

// Slot k (a quad) of the perimeter nodes inside the output rectangle widened by e.
struct EdgeList {
  int ax, bx, ay, by, n_rows, n_cols, n;
  bool px, py;
  __host__ __device__ EdgeList(const TileRect& t, int e, int nx, int ny, bool px_, bool py_) : px(px_), py(py_) {
    ax = px || t.x0 > e ? t.x0 - e : 0;
    bx = px || t.x1 + e < nx ? t.x1 + e : nx;
    ay = py || t.y0 > e ? t.y0 - e : 0;
    by = py || t.y1 + e < ny ? t.y1 + e : ny;
    n_rows = n_cols = n = 0;
    for (int k = 0; k < 4; ++k) {
      const int yk = line(k, ny), xk = line(k, nx);
      if ((k < 2 || py) && yk >= ay && yk < by) n_rows |= 1 << k, n += bx - ax;
      if ((k < 2 || px) && xk >= ax && xk < bx) n_cols |= 1 << k, n += by - ay;
    }
  }
  // the first and last line of an axis, and along a periodic one their images
  static __host__ __device__ int line(int k, int n) { return k == 0 ? 0 : (k == 1 ? n - 1 : (k == 2 ? -1 : n)); }
  // node k < n; false where a column's node already came with its row
  __host__ __device__ bool node(int k, int nx, int ny, int& x, int& y) const {
    for (int c = 0; c < 4; ++c)
      if (n_rows >> c & 1) {
        if (k < bx - ax) {
          x = ax + k;
          y = line(c, ny);
          return true;
        }
        k -= bx - ax;
      }
    for (int c = 0; c < 4; ++c)
      if (n_cols >> c & 1) {
        if (k < by - ay) {
          x = line(c, nx);
          y = ay + k;
          for (int d = 0; d < 4; ++d)
            if ((n_rows >> d & 1) && line(d, ny) == y) return false;
          return true;
        }
        k -= by - ay;
      }
    return false;
  }
};

__device__ __forceinline__ EdgeSlot edge_slot(const EdgeList& list, int u, const TileRegion& reg, const Geom& g,
                                              const Nsbc& p) {
  EdgeSlot s;
  const int q = u & 3;
  s.x = s.y = 0;
  s.any = (u >> 2) < list.n && list.node(u >> 2, g.nx, g.ny, s.x, s.y);
  s.en.x = s.x < 0 ? s.x + g.nx : (s.x >= g.nx ? s.x - g.nx : s.x);
  s.en.y = s.y < 0 ? s.y + g.ny : (s.y >= g.ny ? s.y - g.ny : s.y);
  s.en.nxn = list.px ? 0 : (s.en.x == 0 ? -1 : (s.en.x == g.nx - 1 ? 1 : 0));
  s.en.nyn = list.py ? 0 : (s.en.y == 0 ? -1 : (s.en.y == g.ny - 1 ? 1 : 0));
  s.en.open = s.en.nxn != 0 || s.en.nyn != 0;
  const QuadPair pr = quad_pair(q);
  auto known = [&](int x, int y) {
    return (list.px || (x >= 0 && x < g.nx)) && (list.py || (y >= 0 && y < g.ny));
  };
  s.kp = known(s.x - pr.cx, s.y - pr.cy);
  s.km = known(s.x + pr.cx, s.y + pr.cy);
  s.want = s.en.open && q <= p.order;
  const bool split = p.corner == 1 && s.en.nxn != 0 && s.en.nyn != 0;  // the vertical edge's normal first
  s.at = 9 * (s.y - reg.y0) * reg.w + s.x - reg.x0;
  s.back = s.at - q * (9 * (split ? 0 : s.en.nyn) * reg.w + s.en.nxn);
  return s;
}

// A node's results: to the next state in shared memory, and to device memory
// at the end or where a neighbour tile's halo takes the node.
template <typename T>
struct EdgeDst {
  using C = typename Store<T>::C;
  C* s;  // population 0
  int w;
  T* b;
  long long plane;
  bool to_s, to_b;
  __device__ __forceinline__ void st(int i, int, int, C v) const {
    const T t = Store<T>::cvt(v);
    if (to_s) s[i * w] = Store<T>::ld1s(&t);
    if (to_b) Store<T>::st1(b + i * plane, v);
  }
};

// nsbc_edge_nodes on a node of the region's state src (the same operations in
// the same order); `from` is the state for the second pass of a corner.
template <typename T, int MODEL, bool SHIFT>
__device__ __forceinline__ void tile_edge(const typename Store<T>::C* __restrict__ src, const TileState<T>& from,
                                          int w, const EdgeDst<T>& to, const Geom& g, const Nsbc& p,
                                          const Rates<typename Store<T>::C>& r, const EdgeSlot& s, int q) {
  using C = typename Store<T>::C;
  const unsigned quad = 0xFu << ((threadIdx.x & 31) & ~3);
  const QuadPair pr = quad_pair(q);
  auto ld = [&](int o) { return Store<T>::kScale == 1 ? src[o] : src[o] * C(1.0 / Store<T>::kScale); };
  const C hp = s.kp ? ld(s.at + (pr.ip - 9 * pr.cy) * w - pr.cx) : C(0);
  const C hm = s.km ? ld(s.at + (pr.im + 9 * pr.cy) * w + pr.cx) : C(0);
  const C h0 = ld(s.at);
  C v[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) v[i] = s.want ? ld(s.back + i * w) : C(0);
  const bool corner = s.en.nxn != 0 && s.en.nyn != 0, split = p.corner == 1 && corner;
  Predicted<C> mine =
      quad_predict<T, SHIFT>(v, far_of(r.z), quad, q < 3 ? q : 0, corner && !split, predict_of<C>(p));
  if (split)
    mine = predicted_mean(mine, corner_second_prediction<T, SHIFT>(from, s.en.x, s.en.y - q * s.en.nyn, far_of(r.z),
                                                                  quad, q, predict_of<C>(p)));
  const C mcq = predicted_value(mine);
  C mc[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) mc[c] = __shfl_sync(quad, mcq, c, 4);
  quad_finish<T, MODEL, SHIFT>(to, g, p, r, s.en, pr, q, quad, hp, hm, h0, s.kp, s.km, mc, true);
}

constexpr int kRowSlack = 72;  // elements

// One step of a tile, src -> dst (region states in shared memory), by a block
// of NT threads: computed on the output rectangle widened by e nodes on each
// side (clipped at the domain's edges, running past them along a periodic
// axis).  last: the step's output nodes go to B and nothing to dst.  Sides of
// the rectangle that lie on an edge are at least two nodes deep: the
// second-order difference reads the node two further in.
template <typename T, int MODEL, bool SHIFT, int NT>
__device__ __forceinline__ void tile_step(const typename Store<T>::C* __restrict__ src,
                                          typename Store<T>::C* __restrict__ dst, T* __restrict__ B, const Geom& g,
                                          const Nsbc& p, const Rates<typename Store<T>::C>& r, const TileRect& t,
                                          const TileRegion& reg, int e, bool last) {
  using S = Store<T>;
  using C = typename S::C;
  const int tid = threadIdx.x, w = reg.w, h = reg.h, rx0 = reg.x0, ry0 = reg.y0;
  const bool px = p.periodic_x != 0, py = p.periodic_y != 0;
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
      const TileState<T> to{dst, rx0, ry0, w, g.nx, g.ny, h};
      const GlobalDst<T> out{B, g.plane, g.pitch};
      if (last)
        nsbc_edge_nodes<T, MODEL, 1, SHIFT>(from, out, g, p, r, en, ok, tid & 3);
      else
        nsbc_edge_nodes<T, MODEL, 1, SHIFT>(from, to, g, p, r, en, ok, tid & 3);
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

// One step of a resident tile, as tile_step.  Beside it, the last step of a
// round (e = 0) writes the nodes nearer than `ring` to a side that has a
// neighbour to B as well.  list: the perimeter nodes of the round's widest
// step, `mine` this thread's slot of it.
template <typename T, int MODEL, bool SHIFT, int NT>
__device__ __forceinline__ void resident_step(const typename Store<T>::C* __restrict__ src,
                                              typename Store<T>::C* __restrict__ dst, T* __restrict__ B,
                                              const Geom& g, const Nsbc& p, const Rates<typename Store<T>::C>& r,
                                              const TileRect& t, const TileRegion& reg, int e, bool last, int ring,
                                              const CellConst<float2>& cell, const EdgeList& list,
                                              const EdgeSlot& mine) {
  using S = Store<T>;
  using C = typename S::C;
  const int tid = threadIdx.x, w = reg.w, rx0 = reg.x0, ry0 = reg.y0;
  const bool px = p.periodic_x != 0, py = p.periodic_y != 0;
  const int ax = px ? t.x0 - e : max(t.x0 - e, 0), bx = px ? t.x1 + e : min(t.x1 + e, g.nx);
  const int ay = py ? t.y0 - e : max(t.y0 - e, 0), by = py ? t.y1 + e : min(t.y1 + e, g.ny);
  // output nodes [cx0, cx1) x [cy0, cy1): no neighbour takes them
  const int cx0 = px || t.x0 > 0 ? t.x0 + ring : t.x0, cx1 = px || t.x1 < g.nx ? t.x1 - ring : t.x1;
  const int cy0 = py || t.y0 > 0 ? t.y0 + ring : t.y0, cy1 = py || t.y1 < g.ny ? t.y1 - ring : t.y1;
  auto publish = [&](int x, int y) { return e == 0 && !(x >= cx0 && x < cx1 && y >= cy0 && y < cy1); };
  auto edge = [&](const EdgeSlot& s) {
    if (!s.any || s.x < ax || s.x >= bx || s.y < ay || s.y >= by) return;
    tile_edge<T, MODEL, SHIFT>(src, TileState<T>{const_cast<C*>(src), rx0, ry0, w, g.nx, g.ny, reg.h}, w,
                               EdgeDst<T>{dst + s.at, w, B + (long long)s.en.y * g.pitch + s.en.x, g.plane, !last,
                                          last || publish(s.x, s.y)},
                               g, p, r, s, tid & 3);
  };
#pragma unroll 1
  for (int u = tid; u < 4 * list.n; u += NT) edge(u == tid ? mine : edge_slot(list, u, reg, g, p));
  // interior nodes: the rectangle without the edges of non-periodic axes
  const int ix = px ? ax : max(ax, 1), jx = px ? bx : min(bx, g.nx - 1);
  const int iy = py ? ay : max(ay, 1), jy = py ? by : min(by, g.ny - 1);
  const int wi = max(jx - ix, 0);
  // A warp takes 64 columns of a row, two nodes 32 apart per lane, so that
  // a row costs one address per population; the warps the boundary leaves
  // free take the rows where there are enough of them.  (Lanes past the
  // row read what follows it in shared memory, kRowSlack at the end, and
  // store nothing.)
  constexpr int NW = NT / 32;
  const int lane = tid & 31, busy = (4 * list.n + 31) >> 5, skip = 2 * busy <= NW ? busy : 0;
  const int chunks = (wi + 63) >> 6, tasks = chunks * max(jy - iy, 0);
  const bool pub = e == 0;
  for (int q = (tid >> 5) - skip; q < tasks; q += NW - skip) {
    if (q < 0) break;
    const int chunk = chunks == 1 ? 0 : q / (jy - iy), y = iy + q - chunk * (jy - iy);
    const int x = ix + 64 * chunk + lane;
    const int at = 9 * (y - ry0) * w + (x - rx0);
    float2 f[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const C* o = src + at + (i - 9 * cy(i)) * w - cx(i);
      f[i] = make_float2(o[0], o[32]);
    }
    collide<MODEL, SHIFT>(f, r, C(S::kScale), cell);
    auto inside = [&](int xk) {
      return xk < jx && !(px && (xk == 0 || xk == g.nx - 1 || xk == -1 || xk == g.nx)) &&
             !(py && (y == 0 || y == g.ny - 1 || y == -1 || y == g.ny));
    };
    const bool ok[2] = {inside(x), inside(x + 32)};
    if (!last) {
      C* o = dst + at;
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        if (ok[0]) o[i * w] = stored<T>(f[i].x);
        if (ok[1]) o[i * w + 32] = stored<T>(f[i].y);
      }
    }
    if (last || pub) {  // e = 0: no coordinate lies past the domain
      T* o = B + (long long)y * g.pitch + x;
      const bool out[2] = {ok[0] && (last || publish(x, y)), ok[1] && (last || publish(x + 32, y))};
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        if (out[0]) S::st1r(o + i * g.plane, f[i].x);
        if (out[1]) S::st1r(o + i * g.plane + 32, f[i].y);
      }
    }
  }
  __syncthreads();
}

// `steps` steps of the output nodes `t` (A: step n, B: step n + steps), by a
// block of NT threads: step j is computed on the output rectangle widened by
// steps - j nodes, so the last one needs no other tile's results.
template <typename T, int MODEL, bool SHIFT, int NT>
__device__ __forceinline__ void tile_steps(const T* __restrict__ A, T* __restrict__ B, const Geom& g, const Nsbc& p,
                                           const Rates<typename Store<T>::C>& r, const TileRect& t, int steps,
                                           typename Store<T>::C* smem) {
  const TileRegion reg = tile_region(g.nx, g.ny, p.periodic_x != 0, p.periodic_y != 0, t, steps);
  const int other = 9 * reg.w * reg.h;  // the two steps' states: smem and smem + other
  tile_load<T, NT>(A, g, reg, smem);
  for (int j = 1; j <= steps; ++j)
    tile_step<T, MODEL, SHIFT, NT>(smem + (j & 1 ? 0 : other), smem + (j & 1 ? other : 0), B, g, p, r, t, reg,
                                   steps - j, j == steps);
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
  const CellConst<float2> k = cell_const<MODEL, !SHIFT, float2>(r, float(Store<T>::kScale));
  const T* mine = ring + 2 * lane;
  int slot = 0;
  auto next = [](int sl) { return sl + 1 == R::DEPTH ? 0 : sl + 1; };
  int s = s0;
  // Row `row` has arrived; else the item ends, once the copies still in flight
  // into the ring have (or have been waited for as long again).
  auto wait = [&](int sl, int row) {
    if (__all_sync(0xffffffffu, mbar_wait(&bar[sl], (phase >> sl) & 1u))) {
      phase ^= 1u << sl;
      return true;
    }
    if (lane == 0) atomicExch(&err[2], 1);
    const int last = min(s1, max(s0 + R::DEPTH - 1, row + R::DEPTH - 3));  // newest row staged
    for (; row <= last; ++row, sl = next(sl)) mbar_wait(&bar[sl], (phase >> sl) & 1u);
    return false;
  };
  for (;;) {
    if (K == R::K && s >= s0 + 2 * R::K) {
#pragma unroll 1
      for (; s < s1; s += 2) {
        if (!wait(slot, s)) return false;
        roll_row<true, T, MODEL, SHIFT>(stage, out, g, r, K, x0, s0, s, s1, slot, mine, lo, hi, whole, some, c, k);
        slot = next(slot);
        if (!wait(slot, s + 1)) return false;
        roll_row<true, T, MODEL, SHIFT>(stage, out, g, r, K, x0, s0, s + 1, s1, slot, mine, lo, hi, whole, some, c, k);
        slot = next(slot);
      }
    }
    if (s > s1) break;
    if (!wait(slot, s)) return false;
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
// resets the counters.  A warp whose wait gave up sets sched[2] and takes no
// more items, but counts as out, so the next pass starts from zero again.
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
    if (!roll_item<T, MODEL, SHIFT>(A, B, g, r, steps, strip * R::OUT, Ya, Yb, ring, bar, phase, lane, sched)) break;
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

// The largest piece of a side of n nodes in 1 .. most pieces of 4 or more, and
// the fewest pieces (from three on) that are no larger than those of g.
struct TileCuts {
  int most = 0, size[65], fewest[65];
  explicit TileCuts(int n) {
    for (int g = 1; g <= 64 && n / g >= 4; ++g) {
      size[most = g] = (n + g - 1) / g;
      fewest[g] = g > 3 && size[g] == size[g - 1] ? fewest[g - 1] : g;
    }
  }
};

inline TilePlan plan_tiles(int nx, int ny, bool f64, bool px, bool py, int sms) {
  // microseconds, measured: launch, load per node, step, node, boundary node
  const double t_launch = 2.0, t_load = f64 ? 1.4e-3 : 0.7e-3, t_step = f64 ? 0.9 : 0.35;
  const double t_node = f64 ? 15e-3 : 0.45e-3, t_edge = f64 ? 100e-3 : 3e-3;
  const size_t elt = f64 ? 8 : 4, room = kTileRoom;
  TilePlan best;
  const TileCuts cx(nx), cy(ny);
  for (int steps : {1, 2, 3, 4, 5, 6, 8, 10, 12})
    for (int gx = 1; gx <= cx.most; ++gx) {
      const int tw = cx.size[gx], w = px || gx > 2 ? tw + 2 * steps : (gx == 2 ? tw + steps : tw);
      if (px && w > nx) continue;
      // From three rows of tiles on, more rows in the same number of waves
      // cost less: only the fewest rows with the smallest tiles of 1 .. 8
      // waves can win (a plan then takes tens of microseconds).
      for (int c = -1; c <= 8; ++c) {
        const int top = std::min(cy.most, c * sms / gx);
        if (c > 0 && top < 3) continue;
        const int gy = c <= 0 ? c + 2 : cy.fewest[top];
        if (gy > cy.most || gx * gy > 8 * sms) continue;
        const int waves = (gx * gy + sms - 1) / sms;
        const int th = cy.size[gy], h = py || gy > 2 ? th + 2 * steps : (gy == 2 ? th + steps : th);
        if (py && h > ny) continue;
        const size_t smem = 2 * 9 * (size_t)w * h * elt;
        if (smem > room) continue;
        double block = 0.8 + t_load * w * h;
        // no less than steps on the tile alone: most candidates end here
        if ((t_launch + waves * (block + steps * (t_step + t_node * tw * th + t_edge * std::max(tw, th)))) *
                (1.0 - 1e-9) >
            best.us * steps)
          continue;
        for (int j = 1; j <= steps; ++j) {
          const double c = (double)(steps - j) / steps;  // of the halo that step j still covers
          const double wj = tw + (w - tw) * c, hj = th + (h - th) * c;
          block += t_step + t_node * wj * hj + t_edge * std::max(wj, hj);
        }
        const double us = (t_launch + waves * block) / steps;
        if (us < best.us) best = TilePlan{gx, gy, steps, (int)smem, us};
      }
    }
  return best;
}

// ---------------------------------------------------------------------------
// A domain that stays on chip: gx x gy tiles, a block each, all resident at
// once (cooperative launch), hold the state in shared memory for all the
// steps of a launch.  Every `halo` steps a block writes the nodes its
// neighbours' halos take to device memory, raises its flag, waits for the
// flags of its (up to 8) neighbours and reads its own halo.  Rounds write B
// and A in turn: a block writes a buffer again two rounds later, when every
// neighbour has raised the flag of the round between, so has read the first.
// What bounds it: the boundary nodes' chain of operations, about 1 us a step in
// the blocks that hold an edge, while the others wait for them in the
// exchange, itself 1.6 us a round.  So rounds are long (the halo is computed
// twice rather than exchanged), the boundary's lookups are made once, and its
// warps are left out of the rows.  Microseconds a step against the forms of
// one launch per step or per tile plan: 128^2 channel (MRT) 2.4 against 2.7,
// 320^2 f32 2.6 against 2.9, 613 x 377 f16 3.4 against 3.7.  In double the FP64
// pipe is the bound and the boundary blocks' share of it the longest: 200^2
// 12.5 against 9.1, so it is not built.
// ---------------------------------------------------------------------------
constexpr int kFlagStride = 8;  // a flag per 32 bytes

// The halo of a tile's region (the region without the tile), element by
// element: first the whole rows above and below, then the sides of the rows
// between.
struct TileHalo {
  int w, tw, th, top, left;      // region width, tile, rows above, columns beside
  int cols, n_rows, n;           // columns of a row between; elements of the whole rows, of all
  unsigned mul_w, mul_c;         // e / w and e / cols as high words (exact: e w < 2^32)
  __host__ __device__ TileHalo(const TileRect& t, const TileRegion& reg)
      : w(reg.w), tw(t.x1 - t.x0), th(t.y1 - t.y0), top(t.y0 - reg.y0), left(t.x0 - reg.x0) {
    cols = w - tw;
    n_rows = 9 * (reg.h - th) * w;
    n = n_rows + 9 * th * cols;
    mul_w = 0xffffffffu / (unsigned)w + 1u;
    mul_c = cols > 1 ? 0xffffffffu / (unsigned)cols + 1u : 0u;
  }
  // element e < n: population i of region node (lx, ly)
  __host__ __device__ void at(int e, int& i, int& lx, int& ly) const {
    const bool row = e < n_rows;
    if (!row) e -= n_rows;
    const int k = row || cols > 1 ? (int)((unsigned long long)(unsigned)e * (row ? mul_w : mul_c) >> 32) : e;
    lx = e - k * (row ? w : cols);
    ly = k / 9;
    i = k - 9 * ly;
    if (row) {
      if (ly >= top) ly += th;
    } else {
      if (lx >= left) lx += tw;
      ly += top;
    }
  }
};

// from device memory, past the L1 cache
template <typename T, int NT>
__device__ __forceinline__ void tile_halo(const T* B, const Geom& g, const TileHalo& halo, const TileRegion& reg,
                                          typename Store<T>::C* dst) {
  using S = Store<T>;
  constexpr int Q = 6;  // loads in flight per thread
  for (int e0 = threadIdx.x; e0 < halo.n; e0 += Q * NT) {
    T v[Q];
    int at[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      at[q] = -1;
      if (e0 + q * NT >= halo.n) continue;
      int i, lx, ly;
      halo.at(e0 + q * NT, i, lx, ly);
      at[q] = (9 * ly + i) * reg.w + lx;
      int x = reg.x0 + lx, y = reg.y0 + ly;
      x = x < 0 ? x + g.nx : (x >= g.nx ? x - g.nx : x);
      y = y < 0 ? y + g.ny : (y >= g.ny ? y - g.ny : y);
      const T* src = B + i * g.plane + (long long)y * g.pitch + x;
      v[q] = in_bounds(src, sizeof(T)) ? __ldcg(src) : T(0.f);
    }
#pragma unroll
    for (int q = 0; q < Q; ++q)
      if (at[q] >= 0) dst[at[q]] = S::ld1s(&v[q]);
  }
}

// Whether *flag reaches `want` before `limit` SM clock cycles have passed (it
// is looked at once in any case).  32 bits hold limits up to 4e9 cycles, with
// 0.1 s and more between two looks; in 64 bits the wait cost a resident 128^2
// channel 0.7 % (489 against 485 us for 200 steps).
__device__ __forceinline__ bool flag_wait(const unsigned* flag, unsigned want, unsigned limit) {
  const unsigned t0 = clock();
  for (;;) {
    unsigned seen;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(flag) : "memory");
    if ((int)(seen - want) >= 0) return true;
    if ((unsigned)clock() - t0 >= limit) return false;
  }
}

// flags[block]: rounds whose outer nodes the block has written (zero at
// launch).  A wait that gives up after `limit` cycles sets err[2] and ends its
// block; so, in turn, do the blocks that wait for it.
template <typename T, int MODEL, bool SHIFT>
__global__ void __launch_bounds__(kTileThreads)
    resident_kernel(T* A, T* B, Geom g, Nsbc p, Rates<typename Store<T>::C> r, int gx, int gy, int halo, int steps,
                    unsigned* flags, unsigned limit, int* err) {
  using C = typename Store<T>::C;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  C* smem = reinterpret_cast<C*>(smem_raw);
  const int ty = blockIdx.x / gx, tx = blockIdx.x - ty * gx, tid = threadIdx.x;
  const TileRect t{(int)((unsigned)g.nx * tx / gx), (int)((unsigned)g.ny * ty / gy),
                   (int)((unsigned)g.nx * (tx + 1) / gx), (int)((unsigned)g.ny * (ty + 1) / gy)};
  const bool px = p.periodic_x != 0, py = p.periodic_y != 0;
  const TileRegion reg = tile_region(g.nx, g.ny, px, py, t, halo);
  const int other = 9 * reg.w * reg.h;
  const TileHalo halo_of(t, reg);
  const CellConst<float2> cell = cell_const<MODEL, false, float2>(r, C(Store<T>::kScale));
  const EdgeList list(t, halo - 1, g.nx, g.ny, px, py);
  const EdgeSlot slot = edge_slot(list, tid, reg, g, p);
  // thread k < 9 waits for the neighbour (k % 3 - 1, k / 3 - 1)
  const unsigned* theirs = nullptr;
  if (tid < 9 && tid != 4) {
    int nx = tx + tid % 3 - 1, ny = ty + tid / 3 - 1;
    if (px) nx = nx < 0 ? gx - 1 : (nx == gx ? 0 : nx);
    if (py) ny = ny < 0 ? gy - 1 : (ny == gy ? 0 : ny);
    if (nx >= 0 && nx < gx && ny >= 0 && ny < gy) theirs = flags + (ny * gx + nx) * kFlagStride;
  }
  tile_load<T, kTileThreads>(A, g, reg, smem);
  int at = 0;  // where the newest state is: smem + at
  for (unsigned round = 1;; ++round) {
    const int k = min(halo, steps);
    steps -= k;
    for (int j = 1; j <= k; ++j) {
      resident_step<T, MODEL, SHIFT, kTileThreads>(smem + at, smem + (other - at), round & 1 ? B : A, g, p, r, t, reg,
                                                     k - j, steps == 0 && j == k, halo, cell, list,
                                                     slot);
      at = other - at;
    }
    if (steps == 0) return;
    // the block's stores are ordered before the flag by the step's barrier and this fence
    if (tid == 0) {
      __threadfence();
      asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(flags + blockIdx.x * kFlagStride), "r"(round)
                   : "memory");
    }
    if (__syncthreads_or(theirs && !flag_wait(theirs, round, limit))) {
      if (tid == 0) atomicExch(&err[2], 1);
      return;
    }
    tile_halo<T, kTileThreads>(round & 1 ? B : A, g, halo_of, reg, smem + at);
    __syncthreads();
  }
}

// Host: the tiles and the halo of a resident domain, by a model of a round;
// steps = 0 where the state does not fit the SMs' shared memory.
inline TilePlan plan_resident(int nx, int ny, bool px, bool py, int sms) {
  // microseconds: a round's exchange, halo node, step (the boundary's chain of operations), row of 64 nodes,
  // boundary node (of a corner tile; both lines of a periodic axis)
  const double t_round = 2.6, t_halo = 0.7e-3, t_step = 0.9, t_row = 0.025, t_edge = 0.01;
  TilePlan best;
  for (int halo = 1; halo <= 8; ++halo) {
    const int side = std::max(4, halo);  // a halo reaches no further than the next tile
    for (int gx = 1; gx <= sms && nx / gx >= side; ++gx)
      for (int gy = 1; gx * gy <= sms && ny / gy >= side; ++gy) {
        const int tw = (nx + gx - 1) / gx, th = (ny + gy - 1) / gy;
        const int w = px || gx > 2 ? tw + 2 * halo : (gx == 2 ? tw + halo : tw);
        const int h = py || gy > 2 ? th + 2 * halo : (gy == 2 ? th + halo : th);
        if ((px && w > nx) || (py && h > ny)) continue;
        const size_t smem = tile_bytes<float>(w, h) + kRowSlack * sizeof(float);
        if (smem > kTileRoom) continue;
        double us = t_round + t_halo * ((double)w * h - (double)tw * th);
        // no less than `halo` steps on the tile alone, as in plan_tiles
        if ((us + halo * (t_step + t_row * ((tw + 63) / 64) * th + t_edge * (tw + th))) * (1.0 - 1e-9) > best.us * halo)
          continue;
        for (int j = 1; j <= halo; ++j) {
          const double c = (double)(halo - j) / halo;  // of the halo that step j still covers
          const double wj = tw + (w - tw) * c, hj = th + (h - th) * c;
          const double edge = (px || gx == 1 ? 2 : 1) * hj + (py || gy == 1 ? 2 : 1) * wj;
          us += t_step + t_row * (int)((wj + 63) / 64) * hj + t_edge * edge;
        }
        if (us / halo < best.us) best = TilePlan{gx, gy, halo, (int)smem, us / halo};
      }
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
      break;
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
