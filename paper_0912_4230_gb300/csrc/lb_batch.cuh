// Batched step: many lattices (contexts) advanced by one persistent launch per
// step.
//
// The work list is the concatenation of every lattice's blocks of the
// per-cell step kernel (same block shapes, same warp-to-flux-slot mapping),
// one 64-bit descriptor per block,
// so each lattice computes exactly what its own launch would. The grid is a
// fixed number of resident blocks that walk the list with stride gridDim.x.
// The lattices' arguments travel in the launch's parameter space
// (__grid_constant__), so the per-cell update reads them as constant-bank
// operands, as in the per-cell kernel, rather than from memory.
#pragma once

#include "lb_kernels.cuh"

namespace lbgb {

template <class Real>
struct BatchEntry {
  StepArgs<Real> a;      // arguments of the lattice's step
  unsigned gx, gy, bx;   // its per-cell launch shape: blocks along x and y, threads along x
                         // (linear: gx blocks of STEP_BLOCK threads)
};

// One virtual block of the work list: lattice (bits 0-15) and block index along
// x (16-31), along y (32-47) and z (48-63) of the lattice's per-cell launch; a
// linear launch's block index takes bits 16-47.
__host__ __device__ inline uint64_t batch_item(unsigned d, unsigned bxi, unsigned byi, unsigned bz) {
  return uint64_t(d) | (uint64_t(bxi) << 16) | (uint64_t(byi) << 32) | (uint64_t(bz) << 48);
}

// lattices per launch: the table stays within the 32 KB parameter space
constexpr int BATCH_MAX = 64;
template <class Real>
struct BatchTable {
  BatchEntry<Real> e[BATCH_MAX];
};
static_assert(sizeof(BatchTable<float>) <= 32000 && sizeof(BatchTable<double>) <= 32000,
              "batch table exceeds the kernel parameter space");

// Virtual blocks [vb_begin, vb_end) of the work list; item d - d_begin is
// the table entry of the block's lattice.
template <class S, int KMODE, bool SOLUTE>
__global__ void __launch_bounds__(STEP_BLOCK, step_blocks<typename S::Real>())
    batched_step_kernel(const __grid_constant__ BatchTable<typename S::Real> tab,
                        const uint64_t *__restrict__ work, unsigned d_begin, unsigned vb_begin,
                        unsigned vb_end) {
  using Real = typename S::Real;
  for (unsigned vb = vb_begin + blockIdx.x; vb < vb_end; vb += gridDim.x) {
    const uint64_t w = __ldg(work + vb);
    const BatchEntry<Real> &e = tab.e[unsigned(w & 0xffffu) - d_begin];
    const StepArgs<Real> &a = e.a;
    const unsigned byi = unsigned(w >> 32) & 0xffffu, bz = unsigned(w >> 48);
    const unsigned bxi = a.linear ? unsigned(w >> 16) : unsigned(w >> 16) & 0xffffu;
    const CellIndex c = cell_index(a, bxi, byi, bz, e.gx, e.gy, e.bx, threadIdx.x & (e.bx - 1),
                                   threadIdx.x / e.bx);
    const unsigned x = c.x, y = c.y, z = c.z, n = c.n, warp_gid = c.warp;
    const uint32_t link = (c.in && a.link) ? __ldg(a.link + n) : 0u;
    Real fin_acc = Real(0), fout_acc = Real(0), drho = Real(0), sC = Real(0);
    bool open_face = false;
    if (c.in)
      update_cell<S, KMODE, SOLUTE>(a, x, y, z, n, link, fin_acc, fout_acc, drho, sC, open_face);
    warp_reductions(a, warp_gid, open_face, fin_acc, fout_acc, drho, sC);
  }
}

}  // namespace lbgb
