// Batched step: many lattices (contexts) advanced by one launch per step.
//
// The launch's blocks are the concatenation of every lattice's cells in blocks
// of STEP_BLOCK in the order of n, with the warps and flux slots of the per-cell
// step kernel (cell_index), so each lattice computes exactly what its own launch
// would; one whose launch was tuned to rows with other warps or another order of
// them is not taken in. The grid is a fixed number of resident blocks that walk the
// concatenation with stride gridDim.x. The lattices' arguments and first blocks
// travel in the launch's parameter space (__grid_constant__), and a block finds
// its lattice there from its number alone: everything up to the arguments is
// the same for the whole grid's arithmetic on blockIdx, so the compiler keeps
// it in uniform registers and reads the arguments as constants, as in the
// per-cell kernel. (From a work list in global memory the lattice's index was a
// value of each thread and every argument a load: 24 lattices of 32^3, FP16,
// 47.9 -> 44.1 us a step.)
#pragma once

#include "lb_kernels.cuh"

namespace lbgb {

// lattices per launch: the table stays within the 32 KB parameter space
constexpr int BATCH_MAX = 64;
template <class Real>
struct BatchTable {
  StepArgs<Real> a[BATCH_MAX];     // arguments of the lattices' steps (linear)
  unsigned begin[BATCH_MAX + 1];   // first block of each lattice; of the n-th, the total
  int n;
};
static_assert(sizeof(BatchTable<float>) <= 32000 && sizeof(BatchTable<double>) <= 32000,
              "batch table exceeds the kernel parameter space");

template <class S, int KMODE, bool SOLUTE>
__global__ void __launch_bounds__(STEP_BLOCK, sizeof(typename S::Real) == 8 ? 3 : 6)
    batched_step_kernel(const __grid_constant__ BatchTable<typename S::Real> tab) {
  using Real = typename S::Real;
  const unsigned total = tab.begin[tab.n];
  for (unsigned vb = blockIdx.x; vb < total; vb += gridDim.x) {
    int d = 0;  // the last lattice that begins at or before vb
    for (int step = BATCH_MAX / 2; step > 0; step /= 2)
      if (d + step < tab.n && tab.begin[d + step] <= vb) d += step;
    const StepArgs<Real> &a = tab.a[d];
    const CellIndex c = cell_index(a, vb - tab.begin[d], 0, 0, 0, 0, STEP_BLOCK, threadIdx.x, 0);
    const uint32_t link = (c.in && a.link) ? __ldg(a.link + c.n) : 0u;
    Real fin_acc = Real(0), fout_acc = Real(0), drho = Real(0), sC = Real(0);
    bool open_face = false;
    if (c.in)
      update_cell<S, KMODE, SOLUTE>(a, c.x, c.y, c.z, c.n, link, fin_acc, fout_acc, drho, sC,
                                    open_face);
    warp_reductions(a, c.warp, open_face, fin_acc, fout_acc, drho, sC);
  }
}

}  // namespace lbgb
