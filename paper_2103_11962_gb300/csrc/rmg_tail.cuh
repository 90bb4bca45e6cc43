// Interface of the one-kernel coarse end of the V-cycle (rmg_tail.cu).
#pragma once

#include "rmg_internal.cuh"

namespace rmg {

constexpr int kTailThreads = 1024;
constexpr int kTailLevels = 6;           // levels one launch takes
constexpr int kTailDense = 384;          // unknowns of the coarse solve done inside,
constexpr int kTailAlone = 256;          // and of one that is all there is inside
constexpr int kTailDenseBlock = 48;      // up to here every block solves alone

// Node of a small level: region, position and region sizes (10 bits each) and the node, one
// 16-byte load.
struct alignas(16) NodeInfo {
  int region, ijl, dims, node;
};

// A copy of a shared node: its slot, the number of copies of the group, the group's start in
// gslot and the first eight copies in ascending order (itself among them).
struct alignas(16) TailSlot {
  int node, count, start, pad;
  int copy[8];
};

template <typename VT, typename CT>
struct TailLevel {
  int n_r, nslots;
  const NodeInfo* info;
  const RegionDev* regions;
  const uint8_t *mask, *mult;
  const NodeInfo* coloured;              // info sorted by Gauss-Seidel colour, or null
  int cstart[9];                         // start of every colour in it
  const TailSlot* slots;
  const int* gslot;
  const CT* coef;
  const VT *dinv, *c1, *c2;
  const float* pw;                       // stored transfer weights to the next level, or null
  VT *u, *u2, *b, *r, *y, *d;
};

template <typename VT, typename CT>
struct TailArgs {
  TailLevel<VT, CT> lev[kTailLevels];
  int nlev;                              // the last one is the coarsest level
  int smoother, nu1, nu2, degree;
  VT omega;
  int down, solve, up;                   // parts to run (all three unless the solve is outside)
  // dense coarse solve (see mixed_coarse_solve)
  int nc, refine;
  const int *cu2slot, *cidx, *gid;
  const float* Ainv32;
  const double *A, *Ainv, *cscale;
  double *xc, *cres;
};

// Geometry of a level for the kernel: node positions, in node order and (with colours) sorted by
// Gauss-Seidel colour, and the copies of the shared nodes.
struct TailGeometry {
  DBuf<NodeInfo> info, coloured;
  DBuf<TailSlot> slots;
  int cstart[9] = {};
  void build(Ctx& c, const Level& L, bool colours);
};
// Blocks of the cluster the kernel runs on here (16 or 8), or 0 when none fits.
template <typename VT, typename CT>
int tail_cluster(int dim, int B);
template <typename VT, typename CT>
void tail_launch(int dim, int B, int cluster, bool next, const TailArgs<VT, CT>& args,
                 cudaStream_t st);     // next: as launch_after

}  // namespace rmg
