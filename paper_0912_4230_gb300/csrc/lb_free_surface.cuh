// Free-surface kernels (Section 3 of the paper): liquid-mass exchange,
// stream/collide of liquid and interface cells with the reconstruction of
// populations coming from empty cells, and the re-typing of cells whose
// liquid fraction leaves [0, 1].
//
// One step is two passes over the list of liquid and interface cells and three
// launches over the few cells that convert:
//   fs_mass      liquid-mass exchange, colour-gradient field
//   fs_step      stream/collide; lists the interface cells that fill or empty
//   fs_convert   re-types the listed cells and their neighbours
//   fs_newcell   populations of new interface cells, excess mass
//   fs_finish    receives the excess mass; liquid fraction, the list's upkeep
// Each needs its neighbours' results of the one before. A drop of radius 24
// converts ~100 of its 70 000 cells a step: as passes over all active tiles the
// conversions took 36 us of a 192x192x128 step (of 55 us), as launches over
// lists about 10 us. Over the cells of active tiles (32x1x2) the two passes ran
// 4 500 warps, in which two lanes of five were live, in two rounds of an SM's
// resident warps; over the listed cells they are 2 100 full warps in one round:
// 37.9 -> 32.9 us a step (with a warp per new cell).
#pragma once

#include "lb_kernels.cuh"

namespace lbgb {

static_assert(FS_BLOCK == FS_LIST_BLOCK, "fs_finish scans a tile per block");
static_assert(FS_BLOCK % 32 == 0 && FS_BLOCK >= 27,
              "whole warps per tile, and a thread for each of the 27 tiles around it");
// With FP32 storage the stream/collide pass takes at most 102 registers (20
// warps per SM): a drop of 70 000 cells is 14 warps an SM, and 80 or 128 registers
// were no faster (38.8 / 38.3 / 38.3 us a step with 768 / 640 / 512 threads). FP64
// takes what it needs.
template <class Real>
constexpr unsigned fs_step_blocks() {
  return sizeof(Real) == 4 ? 640 / FS_BLOCK : 1;
}

// Tiles needed by the next step around cell (x, y, z), as a mask over the 27
// tile offsets (bit (dx+1) + 3(dy+1) + 9(dz+1)): the cell's own tile and the
// tiles holding its D3Q19 neighbours. A neighbour lies in another tile only
// when the cell is on that face of its tile; the last tile of a row may be
// partial and ends at the lattice's last cell, whose neighbour across the
// periodic seam lies in the first tile.
template <class Real>
__device__ __forceinline__ unsigned fs_tile_mask(const FsArgs<Real> &s, unsigned x, unsigned y,
                                                 unsigned z) {
  const auto lo = [](unsigned v, unsigned tile) { return v % tile == 0 ? -1 : 0; };
  const auto hi = [](unsigned v, unsigned tile, int n) {
    return v % tile == tile - 1 || v + 1 == unsigned(n) ? 1 : 0;
  };
  const int x0 = lo(x, FS_TX), x1 = hi(x, FS_TX, s.a.nx);
  const int y0 = lo(y, FS_TY), y1 = hi(y, FS_TY, s.a.ny);
  const int z0 = lo(z, FS_TZ), z1 = hi(z, FS_TZ, s.a.nz);
  unsigned m = 0u;
  for (int dz = z0; dz <= z1; ++dz)
    for (int dy = y0; dy <= y1; ++dy)
      for (int dx = x0; dx <= x1; ++dx)
        if (dx * dx + dy * dy + dz * dz <= 2) m |= 1u << ((dx + 1) + 3 * (dy + 1) + 9 * (dz + 1));
  return m;
}

// The list of cells serves FS_EPOCH steps: new interface cells are appended as
// they appear, cells that empty stay as entries without effect, and the last
// step of the epoch builds the list afresh from the cells that are live then,
// row by row of the active tiles (appended cells would scatter a warp's
// accesses ever more). The tiles' list is kept the same way.
__device__ __forceinline__ unsigned fs_epoch(unsigned c) { return c / FS_EPOCH; }
__device__ __forceinline__ bool fs_rebuilds(unsigned c) { return c % FS_EPOCH == FS_EPOCH - 1; }

// Adds tile t to the list of epoch e unless it is there (stamp e + 1).
template <class Real>
__device__ __forceinline__ void fs_add_tile(const FsArgs<Real> &s, unsigned t, unsigned e) {
  if (atomicExch(s.stamp + t, e + 1u) != e + 1u)
    s.tiles[e & 1u][atomicAdd(&s.cnt->n_tiles[e & 1u], 1u)] = t;
}

// The tile at offset k (0 .. 26, as in fs_tile_mask) of tile (bx, by, bz), wrapped.
template <class Real>
__device__ __forceinline__ unsigned fs_tile_near(const FsArgs<Real> &s, unsigned bx, unsigned by,
                                                 unsigned bz, unsigned k) {
  const unsigned mx = (bx + s.ntx + k % 3 - 1) % s.ntx;
  const unsigned my = (by + s.nty + (k / 3) % 3 - 1) % s.nty;
  const unsigned mz = (bz + s.ntz + k / 9 - 1) % s.ntz;
  return mx + s.ntx * (my + s.nty * mz);
}

// Adds the tiles of the block-wide OR of the cells' masks around tile (bx, by,
// bz) (wrapped; every thread of the block calls it) to the list of epoch e, in
// no particular order: a cell's update depends only on the previous step's
// values.
template <class Real>
__device__ __forceinline__ void fs_stamp_tiles(const FsArgs<Real> &s, unsigned bx, unsigned by,
                                               unsigned bz, unsigned mask, unsigned e) {
  __shared__ unsigned block_mask;
  if (threadIdx.x == 0) block_mask = 0u;
  __syncthreads();
  mask = __reduce_or_sync(0xffffffffu, mask);
  if ((threadIdx.x & 31u) == 0 && mask) atomicOr(&block_mask, mask);
  __syncthreads();
  const unsigned k = threadIdx.x;
  if (k < 27 && ((block_mask >> k) & 1u)) fs_add_tile(s, fs_tile_near(s, bx, by, bz, k), e);
  __syncthreads();  // block_mask is reset for the next tile only after every read
}

// The live cells of tile (thread k is cell (k % FS_TX, (k / FS_TX) % FS_TY, k /
// (FS_TX FS_TY)) of it; every thread of the block calls) go to the cell list of
// epoch e, the tiles within one link of them to its tile list.
template <class Real>
__device__ __forceinline__ void fs_scan_tile(const FsArgs<Real> &s, unsigned tile, unsigned e) {
  const unsigned tx = threadIdx.x % FS_TX, ty = (threadIdx.x / FS_TX) % FS_TY,
                 tz = threadIdx.x / (FS_TX * FS_TY);
  const unsigned r = s.by_ntx.div(tile), bx = tile - r * s.ntx, bz = s.by_nty.div(r),
                 by = r - bz * s.nty;
  const unsigned x = bx * FS_TX + tx, y = by * FS_TY + ty, z = bz * FS_TZ + tz;
  const unsigned n = x + s.a.nx * (y + s.a.ny * z);
  bool live = x < unsigned(s.a.nx) && y < unsigned(s.a.ny) && z < unsigned(s.a.nz);
  if (live) live = !(s.a.link && (s.a.link[n] >> 31)) && s.type[n] != CELL_EMPTY;
  fs_stamp_tiles(s, bx, by, bz, live ? fs_tile_mask(s, x, y, z) : 0u, e);
  const unsigned row = __ballot_sync(0xffffffffu, live), lane = threadIdx.x & 31u;
  unsigned at = 0;
  if (lane == 0 && row) at = atomicAdd(&s.cnt->n_cells[e & 1u], unsigned(__popc(row)));
  at = __shfl_sync(0xffffffffu, at, 0);
  if (live) s.cells[at + __popc(row & ((1u << lane) - 1u))] = n;
}

// After initialisation: one block per tile lists the first step's cells.
template <class Real>
__global__ void __launch_bounds__(FS_BLOCK) fs_seed_kernel(const FsArgs<Real> s) {
  fs_scan_tile(s, blockIdx.x, 0u);
}

// cell(n, x, y, z) for the live cells listed for step c, a thread each.
template <class Real, class F>
__device__ __forceinline__ void fs_cell_loop(const FsArgs<Real> &s, unsigned c, F &&cell) {
  const unsigned cnt = s.cnt->n_cells[fs_epoch(c) & 1u];
  for (unsigned i = blockIdx.x * FS_BLOCK + threadIdx.x; i < cnt; i += gridDim.x * FS_BLOCK) {
    const unsigned n = s.cells[i];
    const unsigned yz = s.a.by_nx.div(n), x = n - yz * s.a.nx, z = s.a.by_ny.div(yz),
                   y = yz - z * s.a.ny;
    cell(n, x, y, z);
  }
}

// Flowchart step g, Eqs. eq:massmacro, eq:massevol, eq:deltamass:
// m(x, t+1) = m(x, t) + sum_q w (f~_opp(q)(x + c_q) - f~_q(x)), with w = 1 when
// either cell is liquid, (lambda(x) + lambda(x + c_q))/2 between two
// interface cells, and no exchange with empty or solid cells. The colour
// gradient field is the new liquid mass (it holds 0 in empty cells and wall_rho
// in solid ones from the initialisation and the conversions).
// The types of all neighbours are loaded together, then the populations of
// nine directions at a time, whatever the types (every address is a cell): one
// wait each instead of one per direction (all 36 populations at once, at 128
// registers, were slower: 12.5 instead of 11.4 us).
template <class S>
__global__ void __launch_bounds__(FS_BLOCK, sizeof(typename S::Real) == 4 ? 12 : 6)
    fs_mass_kernel(const FsArgs<typename S::Real> s) {
  using Real = typename S::Real;
  using T = typename S::T;
  const StepArgs<Real> &a = s.a;
  const unsigned c = s.cnt->step;
  {
    // the flags of the cells that the previous step converted; this step's
    // lists start empty (the counts alternate: the previous ones are read here)
    const unsigned last = (c & 1u) ^ 1u, k = s.cnt->n_near[last];
    for (unsigned i = blockIdx.x * FS_BLOCK + threadIdx.x; i < k; i += gridDim.x * FS_BLOCK)
      s.flag[s.near[i]] = 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      s.cnt->now = c;
      s.cnt->n_flag = 0u;
      s.cnt->n_new = 0u;
      s.cnt->n_near[c & 1u] = 0u;
      if (c % FS_EPOCH == 0) {
        s.cnt->n_tiles[(fs_epoch(c) + 1u) & 1u] = 0u;
        s.cnt->n_cells[(fs_epoch(c) + 1u) & 1u] = 0u;
      }
    }
  }
  fs_cell_loop(s, c, [&](unsigned n, unsigned x, unsigned y, unsigned z) {
    const unsigned N = a.N;
    const uint32_t link = a.link ? __ldg(a.link + n) : 0u;
    const uint8_t t = s.type[n];
    const Real lx = s.lam[n];
    Real m = s.m[n];
    if (t == CELL_EMPTY) return;
    const CellGeo g = cell_geo_xyz(x, y, z, a.nx, a.ny, a.nz);
    const T *fin = static_cast<const T *>(a.f_in);
    // directions that exchange, and those to an interface cell
    uint32_t live = 0, face = 0;
    Unroll<1, Q>::run([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      const uint8_t ty = s.type[(long long)n + ahead_delta<q>(g)];
      if (ty != CELL_EMPTY) live |= 1u << q;
      if (ty == CELL_INTERFACE) face |= 1u << q;
    });
    Unroll<1, Q>::run([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      if ((faces_ahead(q) & g.onface & a.f_wall) || ((link >> opp(q)) & 1u)) live &= ~(1u << q);
    });
    if (t != CELL_INTERFACE) face = 0;
    auto part = [&](auto first) {
      constexpr int q0 = decltype(first)::value;
      Real in[9], out[9];
      Unroll<0, 9>::run([&](auto kc) {
        constexpr int k = decltype(kc)::value, q = q0 + k;
        in[k] = S::template ld_f<opp(q)>(fin + size_t(opp(q)) * N + (long long)n + ahead_delta<q>(g));
        out[k] = S::template ld_f<q>(fin + size_t(q) * N + n);
      });
      Unroll<0, 9>::run([&](auto kc) {
        constexpr int k = decltype(kc)::value, q = q0 + k;
        if (!((live >> q) & 1u)) return;
        // the equilibrium weights of q and opp(q) are equal, so deviations subtract
        const Real diff = in[k] - out[k];
        const Real w = ((face >> q) & 1u)
                           ? Real(0.5) * (lx + s.lam[(long long)n + ahead_delta<q>(g)])
                           : Real(1);
        m += w * diff;
      });
    };
    part(std::integral_constant<int, 1>{});
    part(std::integral_constant<int, 10>{});
    s.m[n] = m;
    s.rhohat_w[n] = m;
  });
}

// Flowchart steps f, h, e, i for liquid and interface cells: pull-stream with
// bounce-back and, for populations that would come from an empty cell, Eq.
// equilempty: f_q = f^eq_q + f^eq_opp(q) - f~_opp(q)(x) at gas density 1 and
// the cell's own V' (recovered from its post-collision populations; exact
// without Darcy drag); moments, colour gradient, BGK collision with forcing
// and surface tension; then lambda = m / rho, and the cells that fill or empty
// are flagged and listed. Populations, colour-gradient field and types of the
// neighbours are loaded together; the populations whose source turns out
// empty, solid or a wall are replaced.
template <class S>
__global__ void __launch_bounds__(FS_BLOCK, fs_step_blocks<typename S::Real>())
    fs_step_kernel(const FsArgs<typename S::Real> s) {
  using Real = typename S::Real;
  using T = typename S::T;
  static_assert(std::is_same<T, Real>::value, "free surface: storage in the collision type");
  const StepArgs<Real> &a = s.a;
  const unsigned N = a.N;
  const unsigned c = s.cnt->now;
  if (blockIdx.x == 0 && threadIdx.x == 0) s.cnt->step = c + 1u;  // read by the next step's first pass
  fs_cell_loop(s, c, [&](unsigned n, unsigned x, unsigned y, unsigned z) {
  const uint32_t link = a.link ? __ldg(a.link + n) : 0u;
  const uint8_t t = s.type[n];
  const CellGeo g = cell_geo_xyz(x, y, z, a.nx, a.ny, a.nz);
  const T *__restrict__ fin = static_cast<const T *>(a.f_in);
  T *__restrict__ fout = static_cast<T *>(a.f_out);
  const Real eps = __ldg(a.eps + n);
  Real d[Q];
  Unroll<0, Q>::run([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    d[q] = S::template ld_f<q>(fin + size_t(q) * N + (long long)n + src_delta<q>(g));
  });
  // sources that are empty cells
  uint32_t from_gas = 0;
  Unroll<1, Q>::run([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    if (s.type[(long long)n + src_delta<q>(g)] == CELL_EMPTY) from_gas |= 1u << q;
  });
  FluidCollide<Real> fc;
  fc.F[0] = fc.F[1] = fc.F[2] = Real(0);
  if (a.A != Real(0)) colour_gradient(a.rhohat, n, g, a.f_wall, a.wall_rho, fc.F);
  const Real mass = s.m[n];
  if (t == CELL_EMPTY) return;
  const uint32_t bounce = bounce_mask(link, g.onface & a.f_wall);
  from_gas &= ~bounce;
  if (bounce)
    Unroll<1, Q>::run([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      if ((bounce >> q) & 1u) d[q] = S::template ld_f<opp(q)>(fin + size_t(opp(q)) * N + n);
    });
  // f^eq_q - w_q at gas density 1 and the cell's own V' (time t), formed per
  // direction from u, 1/eps and u.u (a 19-value array held the kernel at 128
  // registers)
  if (from_gas) {
    Real r = Real(0), j0 = Real(0), j1 = Real(0), j2 = Real(0);
    Unroll<0, Q>::run([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      const Real v = S::template ld_f<q>(fin + size_t(q) * N + n);
      r += v;
      if (cx(q)) j0 += Real(cx(q)) * v;
      if (cy(q)) j1 += Real(cy(q)) * v;
      if (cz(q)) j2 += Real(cz(q)) * v;
    });
    const Real ir = Real(1) / (Real(1) + r);
    const Real gu0 = j0 * ir - Real(0.5) * eps * a.G[0];
    const Real gu1 = j1 * ir - Real(0.5) * eps * a.G[1];
    const Real gu2 = j2 * ir - Real(0.5) * eps * a.G[2];
    const Real gie = Real(1) / eps;
    const Real guu = gu0 * gu0 + gu1 * gu1 + gu2 * gu2;
    auto ge = [&](auto qc) {
      constexpr int q = decltype(qc)::value;
      const Real cu = dot_c<q>(gu0, gu1, gu2);
      return wq<Real>(q) * (Real(3) * cu + Real(4.5) * gie * cu * cu - Real(1.5) * gie * guu);
    };
    Unroll<1, Q>::run([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      if ((from_gas >> q) & 1u)
        d[q] = ge(qc) + ge(std::integral_constant<int, opp(q)>{}) -
               S::template ld_f<opp(q)>(fin + size_t(opp(q)) * N + n);
    });
  }
  Real drho = Real(0), j0 = Real(0), j1 = Real(0), j2 = Real(0);
  Unroll<0, Q>::run([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    drho += d[q];
    if (cx(q)) j0 += Real(cx(q)) * d[q];
    if (cy(q)) j1 += Real(cy(q)) * d[q];
    if (cz(q)) j2 += Real(cz(q)) * d[q];
  });
  const Real rho = Real(1) + drho;
  const Real irho = Real(1) / rho;
  const Real V[3] = {j0 * irho, j1 * irho, j2 * irho};
  const Real tau = a.tau;
  const Real nu = (tau - Real(0.5)) * Real(1.0 / 3.0);
  velocity_solve<KM_NONE>(a.kinv, N, n, eps, nu, V, a.G, fc.Vp, fc.Fe);
  fc.drho = drho;
  fc.rho = rho;
  fc.ie = Real(1) / eps;
  fc.uu = fc.Vp[0] * fc.Vp[0] + fc.Vp[1] * fc.Vp[1] + fc.Vp[2] * fc.Vp[2];
  fc.uF = fc.Vp[0] * fc.Fe[0] + fc.Vp[1] * fc.Fe[1] + fc.Vp[2] * fc.Fe[2];
  fc.itau = Real(1) / tau;
  fc.omt = Real(1) - fc.itau;
  fc.pre = rho * (Real(1) - Real(0.5) * fc.itau);
  fc.Fn = sqrt(fc.F[0] * fc.F[0] + fc.F[1] * fc.F[1] + fc.F[2] * fc.F[2]);
  fc.st = (a.A != Real(0)) && fc.Fn > st_threshold<Real>();
  fc.stc = fc.st ? a.A * eps * tau : Real(0);
  fc.iFn = fc.st ? Real(1) / fc.Fn : Real(0);
  fc.fold(Real(1), Real(0));
  // the post-collision density, summed from the stored values in direction
  // order (as the liquid fraction and a filled cell's excess mass need it)
  Real rp = Real(0);
  Unroll<0, Q>::run([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    const Real v = fc.template post<q>(d[q]);
    S::template st_f<q>(fout + size_t(q) * N + n, v);
    rp += v;  // the stored value: FP32 / FP64 storage holds the collision type
  });
  const Real rho_post = Real(1) + rp;
  s.rho_post[n] = rho_post;
  if (a.fields) write_fields(a.fields, N, n, rho, fc.Vp, Real(0), nu);
  // the moments a new interface cell averages: it was empty, so each of its
  // live neighbours pulled from it in this pass
  if (from_gas) {
    s.mom[n] = rho;
    s.mom[size_t(N) + n] = fc.Vp[0];
    s.mom[2 * size_t(N) + n] = fc.Vp[1];
    s.mom[3 * size_t(N) + n] = fc.Vp[2];
  }
  // flowchart step j, candidates: lambda > 1 + 1e-3 fills, lambda < -1e-3 empties
  if (t == CELL_INTERFACE) {
    const Real lam = mass / rho;
    s.lam[n] = mass / rho_post;
    const uint8_t flag = lam > Real(1.001) ? FS_FILL : (lam < Real(-0.001) ? FS_EMPTYING : FS_NONE);
    if (flag) {
      s.flag[n] = flag;
      s.flagged[atomicAdd(&s.cnt->n_flag, 1u)] = n;
    }
  }
  });
}

// Component `axis` of c_q for the direction q = lane (0 beyond Q), from the
// table packed in two bits each.
__device__ __forceinline__ int fs_lane_c(unsigned lane, int axis) {
  constexpr auto pack = [](int ax) constexpr {
    unsigned long long p = 0;
    for (int q = 0; q < Q; ++q)
      p |= (unsigned long long)((ax == 0 ? cx(q) : ax == 1 ? cy(q) : cz(q)) + 1) << (2 * q);
    return p;
  };
  constexpr unsigned long long px = pack(0), py = pack(1), pz = pack(2);
  const unsigned long long p = axis == 0 ? px : axis == 1 ? py : pz;
  return lane < Q ? int((p >> (2 * lane)) & 3u) - 1 : 0;
}

// The neighbour n + c_q of a cell for the direction q = lane of a warp (lane 0:
// the cell itself); there: it exists and is not solid.
struct FsLane {
  unsigned y;
  bool there;
};
template <class Real>
__device__ __forceinline__ FsLane fs_lane(const FsArgs<Real> &s, unsigned n, unsigned x, unsigned y,
                                          unsigned z, unsigned lane) {
  const StepArgs<Real> &a = s.a;
  const int dx = fs_lane_c(lane, 0), dy = fs_lane_c(lane, 1), dz = fs_lane_c(lane, 2);
  const CellGeo g = cell_geo_xyz(x, y, z, a.nx, a.ny, a.nz);
  const unsigned ahead = (dx > 0 ? 2u : 0u) | (dx < 0 ? 1u : 0u) | (dy > 0 ? 8u : 0u) |
                         (dy < 0 ? 4u : 0u) | (dz > 0 ? 32u : 0u) | (dz < 0 ? 16u : 0u);
  FsLane l;
  l.y = n + unsigned((dx > 0 ? g.dxp : (dx < 0 ? g.dxm : 0)) +
                     (dy > 0 ? g.dyp : (dy < 0 ? g.dym : 0)) +
                     (dz > 0 ? g.dzp : (dz < 0 ? g.dzm : 0)));
  l.there = lane < Q && !(ahead & g.onface & a.f_wall) && !(a.link && (a.link[l.y] >> 31));
  return l;
}

// Sets bits of a cell's flag byte; returns the byte before.
template <class Real>
__device__ __forceinline__ unsigned fs_flag_or(const FsArgs<Real> &s, unsigned n, unsigned bits) {
  const unsigned sh = 8u * (n & 3u);
  return (atomicOr(reinterpret_cast<unsigned *>(s.flag) + (n >> 2), bits << sh) >> sh) & 0xffu;
}

// a cell's settled flag: filled, emptied, or neither
__device__ __forceinline__ bool fs_settled(unsigned b) {
  return (b & FS_FILL) || ((b & FS_EMPTYING) && !(b & FS_CANCELLED));
}

// A mask over the directions q of test(y) for the neighbour y = n + c_q, without
// those behind a wall face or solid. All neighbours are read before any is
// used, whatever they are (the wrapped neighbour is always a cell).
template <class F>
__device__ __forceinline__ uint32_t fs_neighbors_that(unsigned n, const CellGeo &g, uint32_t link,
                                                      unsigned f_wall, F &&test) {
  uint32_t m = 0;
  Unroll<1, Q>::run([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    if (test(unsigned((long long)n + ahead_delta<q>(g)))) m |= 1u << q;
  });
  Unroll<1, Q>::run([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    if ((faces_ahead(q) & g.onface & f_wall) || ((link >> opp(q)) & 1u)) m &= ~(1u << q);
  });
  return m;
}

// New cell types, by the cells the step flagged, a warp per flagged cell and a
// lane per direction (few cells, each a chain of dependent loads and atomics:
// as a thread per cell the 18 neighbours' chains ran one after another, 25 us
// a step): an emptying cell next to a filling one is cancelled; filled ->
// liquid, emptied -> empty, empty next to a filled cell -> interface (flagged
// FS_NEWCELL), liquid next to an emptied cell -> interface. Every settled cell
// lists itself and its neighbours. The types are changed in place: only
// flagged cells become liquid or empty, an emptied one is never next to a
// filled one, and the other changes depend on none of them, so no thread
// misreads a type that another has changed.
template <class Real>
__global__ void __launch_bounds__(FS_LIST_BLOCK) fs_convert_kernel(const FsArgs<Real> s) {
  const StepArgs<Real> &a = s.a;
  const unsigned c = s.cnt->now, k = s.cnt->n_flag, lane = threadIdx.x & 31u;
  for (unsigned i = (blockIdx.x * FS_LIST_BLOCK + threadIdx.x) >> 5; i < k;
       i += gridDim.x * FS_LIST_BLOCK >> 5) {
    const unsigned n = s.flagged[i];
    const bool fill = s.flag[n] & FS_FILL;
    // this lane's neighbour n + c_lane (lane 0: the cell itself)
    const unsigned yz = a.by_nx.div(n), x = n - yz * a.nx, z = a.by_ny.div(yz), y = yz - z * a.ny;
    const FsLane l = fs_lane(s, n, x, y, z, lane);
    const unsigned b = l.y;
    const bool there = l.there;
    const unsigned fb = s.flag[b];
    const uint8_t tb = s.type[b];
    if (!fill && __any_sync(0xffffffffu, there && lane > 0 && (fb & FS_FILL))) {
      if (lane == 0) fs_flag_or(s, n, FS_CANCELLED);
      continue;
    }
    bool fresh = false;
    if (lane == 0) {
      s.type[n] = fill ? CELL_LIQUID : CELL_EMPTY;
    } else if (there) {
      fresh = fill && tb == CELL_EMPTY;
      if (fresh || (!fill && tb == CELL_LIQUID)) s.type[b] = CELL_INTERFACE;
    }
    const unsigned was =
        there ? fs_flag_or(s, b, FS_CLAIMED | (fresh ? unsigned(FS_NEWCELL) : 0u)) : 0u;
    const bool first = there && !(was & FS_CLAIMED);
    const unsigned won = __ballot_sync(0xffffffffu, first);
    unsigned at = 0;
    if (lane == 0 && won) at = atomicAdd(&s.cnt->n_near[c & 1u], unsigned(__popc(won)));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (first) s.near[at + __popc(won & ((1u << lane) - 1u))] = b;
    // new cells also from the end of the flagged list (the two are disjoint):
    // the flag of the first to mark it tells which thread lists it
    if (fresh && !(was & FS_NEWCELL)) s.flagged[a.N - 1u - atomicAdd(&s.cnt->n_new, 1u)] = b;
  }
}

// A new interface cell, by a warp (lane q its neighbour and its population in
// direction q; as a thread's serial code the launch took 11 us for a few dozen
// cells): f = f^eq(mean rho, mean V') of its liquid and interface neighbours that
// are not new themselves. Sums run in the order of q.
template <class S>
__device__ __forceinline__ void fs_new_cell(const FsArgs<typename S::Real> &s, unsigned n,
                                            unsigned lane, unsigned e, bool rebuilds) {
  using Real = typename S::Real;
  const StepArgs<Real> &a = s.a;
  const unsigned N = a.N, all = 0xffffffffu;
  const unsigned yz = a.by_nx.div(n), x = n - yz * a.nx, z = a.by_ny.div(yz), y = yz - z * a.ny;
  const FsLane l = fs_lane(s, n, x, y, z, lane);
  // density and V' of each neighbour as its collision in this step left them
  // (its post-collision populations carry the same moments: the collision
  // conserves mass, and without Darcy drag their momentum is rho (V' + eps G / 2))
  const Real m0 = s.mom[l.y], m1 = s.mom[size_t(N) + l.y], m2 = s.mom[2 * size_t(N) + l.y],
             m3 = s.mom[3 * size_t(N) + l.y];
  const bool in = l.there && lane > 0 && s.type[l.y] != CELL_EMPTY && !(s.flag[l.y] & FS_NEWCELL);
  const unsigned old = __ballot_sync(all, in);
  Real rs = Real(0), u0 = Real(0), u1 = Real(0), u2 = Real(0);
  for (unsigned b = old; b; b &= b - 1u) {
    const int q = __ffs(b) - 1;
    rs += __shfl_sync(all, m0, q);
    u0 += __shfl_sync(all, m1, q);
    u1 += __shfl_sync(all, m2, q);
    u2 += __shfl_sync(all, m3, q);
  }
  const int cnt = __popc(old);
  const Real ic = Real(1) / Real(cnt > 0 ? cnt : 1);
  const Real r = cnt > 0 ? rs * ic : Real(1);
  const Real u[3] = {u0 * ic, u1 * ic, u2 * ic};
  const Real eps = a.eps[n];
  const Real ie = Real(1) / eps, uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  const int dx = fs_lane_c(lane, 0), dy = fs_lane_c(lane, 1), dz = fs_lane_c(lane, 2);
  const Real cu = Real(dx) * u[0] + Real(dy) * u[1] + Real(dz) * u[2];
  const Real w = lane == 0 ? wq<Real>(0) : (dx * dx + dy * dy + dz * dz == 1 ? wq<Real>(5) : wq<Real>(1));
  const Real dev =
      w * ((r - Real(1)) + r * (Real(3) * cu + Real(4.5) * ie * cu * cu - Real(1.5) * ie * uu));
  if (lane < Q) static_cast<typename S::T *>(a.f_out)[size_t(lane) * N + n] = dev;
  Real rp = Real(0);
  for (int q = 0; q < Q; ++q) rp += __shfl_sync(all, dev, q);
  if (lane == 0) {
    // it joins the cell list, unless it emptied in this epoch and is listed
    if (!rebuilds && s.rho_post[n] != fs_mark(e, Real(0)))
      s.cells[atomicAdd(&s.cnt->n_cells[e & 1u], 1u)] = n;
    s.rho_post[n] = Real(1) + rp;  // the density of the stored populations, for lambda
    if (a.fields) write_fields(a.fields, N, n, r, u, Real(0), (a.tau - Real(0.5)) / Real(3));
  }
  // the tiles within one link of it join the tile list
  const unsigned mask = fs_tile_mask(s, x, y, z);
  if ((mask >> lane) & 1u)
    fs_add_tile(s, fs_tile_near(s, x / FS_TX, y / FS_TY, z / FS_TZ, lane),
                rebuilds ? e + 1u : e);
}

// New interface cells take f = f^eq(mean rho, mean V') of their liquid and
// interface neighbours that are not new themselves (hydrodynamic
// equilibrium, no mass); filled and emptied cells hand their excess mass (m -
// rho, or m) in equal shares to the neighbours that are interface cells after
// the re-typing (they keep it when there are none). The share waits in the
// converted cell's liquid fraction, which only interface cells use; an emptied
// cell's density, which only liquid and interface cells use, notes the epoch.
// The tiles around new interface cells join the tile list (the next one when
// this step builds it).
template <class S>
__global__ void __launch_bounds__(FS_LIST_BLOCK) fs_newcell_kernel(const FsArgs<typename S::Real> s) {
  using Real = typename S::Real;
  using T = typename S::T;
  const StepArgs<Real> &a = s.a;
  const unsigned N = a.N;
  const unsigned c = s.cnt->now;
  if (!(blockIdx.x & 1u)) {  // the even blocks take the new cells
    const unsigned lane = threadIdx.x & 31u, k = s.cnt->n_new, e = fs_epoch(c);
    for (unsigned i = ((blockIdx.x >> 1) * FS_LIST_BLOCK + threadIdx.x) >> 5; i < k;
         i += (gridDim.x >> 1) * FS_LIST_BLOCK >> 5)
      fs_new_cell<S>(s, s.flagged[N - 1u - i], lane, e, fs_rebuilds(c));
    return;
  }
  const unsigned k = s.cnt->n_flag;
  for (unsigned i = (blockIdx.x >> 1) * FS_LIST_BLOCK + threadIdx.x; i < k;
       i += (gridDim.x >> 1) * FS_LIST_BLOCK) {
  const unsigned n = s.flagged[i];
  const uint32_t link = a.link ? a.link[n] : 0u;
  const CellGeo g = cell_geo(n, a.nx, a.ny, a.nz);
  const unsigned f = s.flag[n];
  if (!fs_settled(f)) continue;  // cancelled
  const int cnt = __popc(fs_neighbors_that(
      n, g, link, a.f_wall, [&](unsigned y) { return s.type[y] == CELL_INTERFACE; }));
  // a filled cell keeps m = rho: its post-collision density in the collision
  // type (the exported field is float)
  Real share = Real(0);
  if (cnt > 0) {
    const Real m = s.m[n];
    const Real excess = (f & FS_FILL) ? m - s.rho_post[n] : m;
    share = excess / Real(cnt);
    s.m[n] = m - excess;
  }
  s.lam[n] = share;
  if (!(f & FS_FILL)) {  // emptied; its entry in this epoch's list stays
    zero_fields(s.fields, N, n);
    s.rhohat_w[n] = Real(0);
    s.rho_post[n] = fs_mark(fs_epoch(c), Real(0));
  }
  }
}

// Excess mass arrives at the interface cells near a conversion; their lambda =
// m / rho. The last step of an epoch builds both lists.
template <class S>
__global__ void __launch_bounds__(FS_LIST_BLOCK) fs_finish_kernel(const FsArgs<typename S::Real> s) {
  using Real = typename S::Real;
  const StepArgs<Real> &a = s.a;
  const unsigned c = s.cnt->now, k = s.cnt->n_near[c & 1u];
  const unsigned e = fs_epoch(c) + (fs_rebuilds(c) ? 1u : 0u);
  for (unsigned i = blockIdx.x * FS_LIST_BLOCK + threadIdx.x; i < k; i += gridDim.x * FS_LIST_BLOCK) {
    const unsigned n = s.near[i];
    const uint8_t t = s.type[n];
    const uint32_t link = a.link ? a.link[n] : 0u;
    const unsigned yz = a.by_nx.div(n), x = n - yz * a.nx, z = a.by_ny.div(yz), y = yz - z * a.ny;
    const CellGeo g = cell_geo_xyz(x, y, z, a.nx, a.ny, a.nz);
    Real m = s.m[n];
    const Real rho_post = s.rho_post[n];
    const uint32_t from = fs_neighbors_that(n, g, link, a.f_wall,
                                            [&](unsigned y) { return fs_settled(s.flag[y]); });
    if (t != CELL_INTERFACE) continue;
    Unroll<1, Q>::run([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      if ((from >> q) & 1u) m += s.lam[(long long)n + ahead_delta<q>(g)];
    });
    s.m[n] = m;
    s.lam[n] = m / rho_post;
  }
  if (fs_rebuilds(c)) {
    const uint32_t *list = s.tiles[fs_epoch(c) & 1u];
    const unsigned tiles = s.cnt->n_tiles[fs_epoch(c) & 1u];
    for (unsigned i = blockIdx.x; i < tiles; i += gridDim.x) fs_scan_tile(s, list[i], e);
  }
}

}  // namespace lbgb
