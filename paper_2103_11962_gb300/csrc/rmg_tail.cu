// The coarse end of a V-cycle in one kernel.
//
// The coarse levels hold a few thousand nodes each. As separate launches a sweep over such a
// level (two launches) costs 6 to 8 us, nearly all of it launch gaps, ramp-up and the latency of
// one chain of loads, and the dense coarse solve is another chain of about a dozen launches:
// most of the time of a small solve, and still a fifth of a cycle at a million unknowns. Here
// one thread-block cluster (16 blocks of 1024 threads on 16 SMs, 8 where 16 do not fit) runs
// smoothing, residual, restriction, coarse solve, prolongation and post-smoothing of all levels
// that are small enough; the phases are separated by the hardware's cluster barrier instead of
// kernel boundaries. Larger levels need the whole GPU and stay with their own launches
// (tail_levels() in rmg_hier.cu has the rule).
//
// Arrays that one phase writes and a later one reads are read through ordinary loads after the
// barrier's acquire; only coefficients and geometry, which no phase writes, use read-only loads.
#include <cooperative_groups.h>

#include <algorithm>
#include <vector>

#include "rmg_cluster.h"
#include "rmg_kernels.cuh"
#include "rmg_tail.cuh"

namespace rmg {
namespace {

__global__ void k_node_info(Grid G, NodeInfo* __restrict__ info) {
  RMG_FOR_NODES(G)
    int i, j, l;
    decode(li, R, i, j, l);
    info[n] = NodeInfo{tile_.region, i | (j << 10) | (l << 20), R.nx | (R.ny << 10) | (R.nz << 20),
                       n};
  RMG_END_FOR_NODES
}

__global__ void k_tail_slots(int nslots, const int* __restrict__ sgrp,
                             const int* __restrict__ gptr, const int* __restrict__ gslot,
                             TailSlot* __restrict__ slots) {
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nslots; q += gridDim.x * blockDim.x) {
    const int a = gptr[sgrp[q]], e = gptr[sgrp[q] + 1];
    TailSlot t{gslot[q], e - a, a, 0, {}};
    for (int k = 0; k < 8; ++k) t.copy[k] = a + k < e ? gslot[a + k] : t.node;
    slots[q] = t;
  }
}

// What a sweep does with its rows, in two steps: get() reads what the update needs besides the
// row, before the row is formed, so that those loads are in flight with the row's; put() stores
// the update. The arithmetic is that of the epilogues in rmg_kernels.cuh. (One sweep with the
// kind as a run-time value makes a smaller kernel, but its calls and run-time selects cost more
// than the instruction fetches they save: 2374 against 2170 us for the small 2D solve.)
enum TailOp : int { OP_STORE, OP_RESID_SCALED, OP_RESID_ZERO, OP_JACOBI, OP_CHEB0, OP_CHEB };

template <int OP, typename T>
struct TailUpdate {
  T* out;
  const T* b;
  const T* u;
  const T* dinv;
  T* d;
  T c1, c2;
  struct V { T b, u, dinv, d; };
  __device__ __forceinline__ V get(int n) const {
    V v{};
    if (OP != OP_STORE) v.b = b[n];
    if (OP >= OP_JACOBI) {
      v.u = u[n];
      v.dinv = __ldg(dinv + n);
    }
    if (OP == OP_CHEB) v.d = d[n];
    return v;
  }
  __device__ __forceinline__ void put(int n, const V& v, T au, int m) const {
    if (OP == OP_STORE) {
      out[n] = au;
      return;
    }
    const T r = v.b - au;
    if (OP == OP_RESID_SCALED) {
      out[n] = r * inv_mult<T>(m);
    } else if (OP == OP_RESID_ZERO) {
      out[n] = r;
      d[n] = T(0);
    } else if (OP == OP_JACOBI) {
      out[n] = fma(c2 * v.dinv, r, v.u);
    } else {
      const T dn = OP == OP_CHEB0 ? (v.dinv * r) * c2 : c1 * v.d + (c2 * v.dinv) * r;
      d[n] = dn;
      out[n] = v.u + dn;
    }
  }
};

template <int DIM, int B, typename VT, typename CT>
struct Tail {
  static constexpr int KIND = DIM == 3 ? 27 : 9;
  using S = Sten<KIND>;
  using Lev = TailLevel<VT, CT>;
  const TailArgs<VT, CT>& A;
  int tid, nth;

  __device__ void sync() { cooperative_groups::this_cluster().sync(); }

  static __device__ __forceinline__ NodeInfo load_info(const NodeInfo* info, int n) {
    const int4 v = __ldg(reinterpret_cast<const int4*>(info) + n);
    return NodeInfo{v.x, v.y, v.z, v.w};
  }

  // rows of node n: the products of k_stencil / k_bstencil in the same order. A scalar row reads
  // all its coefficients and values before the products and without branches (a neighbour
  // outside the region: the node itself, not used), so that they are in flight together.
  __device__ __forceinline__ void row(const Lev& L, const VT* u, int n, const NodeInfo& I,
                                      VT (&au)[B]) {
    const int i = I.ijl & 1023, j = (I.ijl >> 10) & 1023, l = I.ijl >> 20;
    const int nx = I.dims & 1023, ny = (I.dims >> 10) & 1023, nz = I.dims >> 20;
    const int sy = nx, sz = nx * ny;
    auto inside = [&](int s) {
      const int dx = S::dx(s), dy = S::dy(s), dz = S::dz(s);
      bool ok = true;
      if (dx < 0) ok &= (i > 0);
      if (dx > 0) ok &= (i < nx - 1);
      if (dy < 0) ok &= (j > 0);
      if (dy > 0) ok &= (j < ny - 1);
      if (dz < 0) ok &= (l > 0);
      if (dz > 0) ok &= (l < nz - 1);
      return ok;
    };
    auto offset = [&](int s) { return S::dx(s) + S::dy(s) * sy + S::dz(s) * sz; };
#pragma unroll
    for (int c = 0; c < B; ++c) au[c] = VT(0);
    if (B == 1) {
      CT cf[S::S];
      VT uv[S::S];
#pragma unroll
      for (int s = 0; s < S::S; ++s) cf[s] = __ldg(L.coef + (size_t)s * L.n_r + n);
#pragma unroll
      for (int s = 0; s < S::S; ++s) uv[s] = u[inside(s) ? n + offset(s) : n];
#pragma unroll
      for (int s = 0; s < S::S; ++s) au[0] = inside(s) ? fma(VT(cf[s]), uv[s], au[0]) : au[0];
      return;
    }
#pragma unroll
    for (int s = 0; s < S::S; ++s) {
      if (!inside(s)) continue;
      const int nb = n + offset(s);
      VT uv[B];
#pragma unroll
      for (int c = 0; c < B; ++c) uv[c] = u[(size_t)c * L.n_r + nb];
#pragma unroll
      for (int c = 0; c < B; ++c)
#pragma unroll
        for (int c2 = 0; c2 < B; ++c2)
          au[c] = fma(VT(__ldg(L.coef + ((size_t)(c * B + c2) * S::S + s) * L.n_r + n)), uv[c2],
                      au[c]);
    }
  }

  // interface sums of y, then the epilogue at every copy; the copies of a group are in the slot
  // itself, so their values are read together instead of one after the other
  template <class Epi>
  __device__ void groups(const Lev& L, const Epi& epi) {
    if (!L.nslots) return;
    for (int q = tid; q < B * L.nslots; q += nth) {
      const int c = B == 1 ? 0 : q / L.nslots, s = B == 1 ? q : q - c * L.nslots;
      const int4* t = reinterpret_cast<const int4*>(L.slots + s);
      const int4 h = __ldg(t), k0 = __ldg(t + 1), k1 = __ldg(t + 2);
      const int k[8] = {k0.x, k0.y, k0.z, k0.w, k1.x, k1.y, k1.z, k1.w};
      const VT* y = L.y + (size_t)c * L.n_r;
      const typename Epi::V v = epi.get(c * L.n_r + h.x);
      VT yv[8];
#pragma unroll
      for (int m = 0; m < 8; ++m) yv[m] = m < 2 || m < h.y ? y[k[m]] : VT(0);
      VT sum = VT(0);
#pragma unroll
      for (int m = 0; m < 8; ++m)
        if (m < h.y) sum += yv[m];
      for (int m = 8; m < h.y; ++m) sum += y[__ldg(L.gslot + h.z + m)];
      epi.put(c * L.n_r + h.x, v, sum, h.y);
    }
    sync();
  }

  template <class Epi>
  __device__ void sweep(const Lev& L, const VT* u, const Epi& epi) {
    for (int n = tid; n < L.n_r; n += nth) {
      const NodeInfo I = load_info(L.info, n);
      const bool shared = __ldg(L.mult + n) > 1;
      typename Epi::V v[B];
#pragma unroll
      for (int c = 0; c < B; ++c) v[c] = epi.get(c * L.n_r + n);
      VT au[B];
      row(L, u, n, I, au);
#pragma unroll
      for (int c = 0; c < B; ++c) {
        if (shared) L.y[(size_t)c * L.n_r + n] = au[c];
        else epi.put(c * L.n_r + n, v[c], au[c], 1);
      }
    }
    sync();
    groups(L, epi);
  }

  __device__ void smooth(const Lev& L, VT*& cur, VT*& oth, int nu, bool from_zero, bool post) {
    auto flip = [&] { VT* t = cur; cur = oth; oth = t; };
    const int n = B * L.n_r;
    if (A.smoother == RMG_SMOOTHER_GS) {
      constexpr int ncol = DIM == 3 ? 8 : 4;
      for (int s = 0; s < nu; ++s) {
        if (s == 0 && from_zero) {
          for (int k = tid; k < n; k += nth) {
            L.r[k] = L.b[k];
            L.d[k] = VT(0);
            cur[k] = VT(0);
          }
          sync();
        } else {
          sweep(L, cur, TailUpdate<OP_RESID_ZERO, VT>{L.r, L.b, nullptr, nullptr, L.d, VT(0), VT(0)});
        }
        for (int k = 0; k < ncol; ++k) {
          const int colour = post ? ncol - 1 - k : k;
          for (int q = L.cstart[colour] + tid; q < L.cstart[colour + 1]; q += nth) {
            const NodeInfo I = load_info(L.coloured, q);
            const int m = I.node;
            const VT r = L.r[m], dv = __ldg(L.dinv + m), um = cur[m];
            VT au[B];
            row(L, L.d, m, I, au);
            const VT d = A.omega * (r - au[0]) * dv;
            L.d[m] = d;
            cur[m] = um + d;
          }
          sync();
        }
      }
      return;
    }
    for (int a = 0; a < nu; ++a) {
      const bool zero = a == 0 && from_zero;
      if (A.smoother == RMG_SMOOTHER_JACOBI) {
        if (zero) {
          for (int k = tid; k < n; k += nth) oth[k] = (A.omega * L.dinv[k]) * L.b[k];
          sync();
        } else {
          sweep(L, cur, TailUpdate<OP_JACOBI, VT>{oth, L.b, cur, L.dinv, nullptr, VT(0), A.omega});
        }
        flip();
        continue;
      }
      if (zero) {
        const VT c = L.c2[0];
        for (int k = tid; k < n; k += nth) {
          const VT dn = (L.dinv[k] * L.b[k]) * c;
          L.d[k] = dn;
          oth[k] = dn;
        }
        sync();
      } else {
        sweep(L, cur, TailUpdate<OP_CHEB0, VT>{oth, L.b, cur, L.dinv, L.d, VT(0), L.c2[0]});
      }
      flip();
      for (int k = 1; k < A.degree; ++k) {
        sweep(L, cur, TailUpdate<OP_CHEB, VT>{oth, L.b, cur, L.dinv, L.d, L.c1[k], L.c2[k]});
        flip();
      }
    }
  }

  static constexpr int kSupport = DIM == 3 ? 125 : 25;   // fine nodes a coarse node gathers from

  // linear weights of the support points, in shared memory (their products in FP64 would cost
  // more than the sums)
  static __device__ void fill_weights(VT* wtab) {
    for (int p = threadIdx.x; p < kSupport; p += blockDim.x)
      wtab[p] = VT((DIM == 3 ? w1d(p / 25 - 2) : 1.0) * (w1d((p / 5) % 5 - 2) * w1d(p % 5 - 2)));
    __syncthreads();
  }

  // FP32 weight of fine node f at offset a along `axis` from the stored weights
  static __device__ __forceinline__ float stored(const Lev& F, int f, int axis, int a) {
    const float w = F.pw[(size_t)axis * F.n_r + f];
    return a == 0 ? 1.f : (a > 0 ? 1.f - w : w);
  }

  // b of C = restriction of r of F: a warp per coarse node, a lane per support point (four
  // rounds in 3D); a point outside the region reads the coarse node's own fine node, unused
  __device__ void restrict_to(const Lev& F, const Lev& C, const VT* wtab) {
    constexpr int M = (kSupport + 31) / 32;
    const int lane = tid & 31;
    for (int q = tid >> 5; q < B * C.n_r; q += nth >> 5) {
      const int c = B == 1 ? 0 : q / C.n_r, n = q - c * C.n_r;
      const NodeInfo I = load_info(C.info, n);
      const bool masked = __ldg(C.mask + n) != 0, shared = __ldg(C.mult + n) > 1;
      const RegionDev R = F.regions[I.region];
      const int X = 3 * (I.ijl & 1023), Y = 3 * ((I.ijl >> 10) & 1023);
      const int Z = DIM == 3 ? 3 * (I.ijl >> 20) : 0;
      const int f0 = R.off + X + R.nx * (Y + R.ny * Z);
      const VT* rs = F.r + (size_t)c * F.n_r;
      VT v[M], w[M];
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const int p = 32 * m + lane;
        const int da = p % 5 - 2, db = (p / 5) % 5 - 2, dc = DIM == 3 ? p / 25 - 2 : 0;
        const bool ok = p < kSupport && X + da >= 0 && X + da < R.nx && Y + db >= 0 &&
                        Y + db < R.ny && Z + dc >= 0 && Z + dc < R.nz;
        const int f = ok ? f0 + da + R.nx * (db + R.ny * dc) : f0;
        v[m] = rs[f];
        w[m] = ok ? wtab[p] : VT(0);
        if (F.pw && ok) {
          float ws = stored(F, f, 1, db) * stored(F, f, 0, da);
          if (DIM == 3) ws = stored(F, f, 2, dc) * ws;
          w[m] = VT(ws);
        }
        if (!ok) v[m] = VT(0);
      }
      VT acc = VT(0);
#pragma unroll
      for (int m = 0; m < M; ++m) acc = fma(w[m], v[m], acc);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) (shared ? C.y : C.b)[(size_t)c * C.n_r + n] = masked ? VT(0) : acc;
    }
    sync();
    groups(C, TailUpdate<OP_STORE, VT>{C.b, nullptr, nullptr, nullptr, nullptr, VT(0), VT(0)});
  }

  // u of F += P ubar (as k_prolong, k_prolong_w)
  __device__ void prolong(const Lev& F, VT* u, const Lev& C, const VT* ubar) {
    for (int q = tid; q < B * F.n_r; q += nth) {
      const int c = B == 1 ? 0 : q / F.n_r, n = B == 1 ? q : q - c * F.n_r;
      if (__ldg(F.mask + n)) continue;
      const NodeInfo I = load_info(F.info, n);
      const int i = I.ijl & 1023, j = (I.ijl >> 10) & 1023, l = I.ijl >> 20;
      const RegionDev R = C.regions[I.region];
      const int cx = i / 3, rx = i - 3 * cx, cy = j / 3, ry = j - 3 * cy;
      const int cz = DIM == 3 ? l / 3 : 0, rz = DIM == 3 ? l - 3 * cz : 0;
      const int sy = R.nx, sz = R.nx * R.ny;
      const int dx = cx + 1 < R.nx ? 1 : 0, dy = cy + 1 < R.ny ? sy : 0;
      const int dz = (DIM == 3 && cz + 1 < R.nz) ? sz : 0;
      const VT* b0 = ubar + (size_t)c * C.n_r + R.off + cx + sy * cy + sz * cz;
      VT w[3] = {rem_weight<VT>(rx), rem_weight<VT>(ry), rem_weight<VT>(rz)};
      if (F.pw) {
        w[0] = VT(rx ? F.pw[n] : 0.f);
        w[1] = VT(ry ? F.pw[(size_t)F.n_r + n] : 0.f);
        w[2] = VT(DIM == 3 && rz ? F.pw[(size_t)2 * F.n_r + n] : 0.f);
      }
      auto xline = [&](const VT* p) { return fma(w[0], p[dx], (VT(1) - w[0]) * p[0]); };
      VT acc = fma(w[1], xline(b0 + dy), (VT(1) - w[1]) * xline(b0));
      if (DIM == 3) {
        const VT a1 = fma(w[1], xline(b0 + dz + dy), (VT(1) - w[1]) * xline(b0 + dz));
        acc = fma(w[2], a1, (VT(1) - w[2]) * acc);
      }
      u[(size_t)c * F.n_r + n] += acc;
    }
    sync();
  }

  // x = Abar^-1 rc on the coarsest level and its copies. Every block keeps the right-hand side,
  // the iterate and the scaled FP32 input in its own shared memory and forms them alone (the
  // vectors are short). The rows of the matrix products are spread over the cluster's warps, or,
  // for a small matrix (SOLO), every block computes all of them and waits for no other.
  template <bool SOLO>
  __device__ void coarse_dense(const Lev& L, double* rc, double* v, double* res, float* w,
                               unsigned* red, double* pow2, int nd) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwid = blockDim.x >> 5;
    const int warp = SOLO ? wid : tid >> 5, nwarps = SOLO ? nwid : nth >> 5;
    // w = FP32(s .* src * 2^-e), 2^e near max |s_i src_i| (k_scale_vec32). The largest exponent
    // is found on the integer pipe: an FP64 instruction of all warps takes 512 clocks here.
    auto scale = [&](const double* src) {
      unsigned m = 0;
      for (int i = threadIdx.x; i < nd; i += blockDim.x)
        m = max(m, ((unsigned)__double2hiint(A.cscale[i] * src[i]) >> 20) & 2047u);
      m = __reduce_max_sync(0xffffffffu, m);
      if (lane == 0) red[wid] = m;
      __syncthreads();
      m = __reduce_max_sync(0xffffffffu, red[lane]);
      // biased exponent of 2^e (zero, infinite and NaN inputs: e = 0), at most 2^1022
      const unsigned f = m == 0 || m == 2047 ? 1023u : min(m, 2045u);
      const double p = __hiloint2double((int)((2046u - f) << 20), 0);
      if (threadIdx.x == 0) pow2[0] = __hiloint2double((int)(f << 20), 0);
      for (int i = threadIdx.x; i < nd; i += blockDim.x)
        w[i] = (float)(A.cscale[i] * src[i] * p);
      __syncthreads();
    };
    // row products: eight lanes a row, four rows a warp
    const int sub = lane & 7, quarter = lane >> 3;
    auto dot64 = [&](const double* M, int i, const double* x) {
      double s = 0.0;
      if (i < nd) {
        const double* r = M + (size_t)i * nd;
#pragma unroll 4
        for (int j = sub; j < nd; j += 8) s = fma(__ldg(r + j), x[j], s);
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      return s;
    };
    // after a product: its result, written by all blocks to `part`, in this block's `all`
    auto collect = [&](const double* part, double* all) {
      if (SOLO) {
        __syncthreads();
        return;
      }
      sync();
      for (int i = threadIdx.x; i < nd; i += blockDim.x) all[i] = part[i];
      __syncthreads();
    };
    double* xo = SOLO ? v : A.xc;
    double* ro = SOLO ? res : A.cres;
    // v (+)= s .* (Ainv32 w) * back
    auto gemv32 = [&](bool add) {
      for (int i0 = 4 * warp; i0 < nd; i0 += 4 * nwarps) {
        const int i = i0 + quarter;
        float acc = 0.f;
        if (i < nd) {
          const float* r = A.Ainv32 + (size_t)i * nd;
#pragma unroll 4
          for (int j = sub; j < nd; j += 8) acc = fmaf(__ldg(r + j), w[j], acc);
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (i < nd && sub == 0)
          xo[i] = (add ? v[i] : 0.0) + A.cscale[i] * ((double)acc * pow2[0]);
      }
      collect(A.xc, v);
    };
    for (int k = threadIdx.x; k < nd; k += blockDim.x)
      rc[k] = double(L.b[(size_t)(k % B) * L.n_r + A.cu2slot[k / B]]);
    __syncthreads();
    if (A.refine == 0) {
      for (int i0 = 4 * warp; i0 < nd; i0 += 4 * nwarps) {
        const double s = dot64(A.Ainv, i0 + quarter, rc);
        if (i0 + quarter < nd && sub == 0) xo[i0 + quarter] = s;
      }
      collect(A.xc, v);
      return;
    }
    scale(rc);
    gemv32(false);
    for (int k = 0; k < A.refine; ++k) {
      for (int i0 = 4 * warp; i0 < nd; i0 += 4 * nwarps) {
        const int i = i0 + quarter;
        const double s = dot64(A.A, i, v);
        if (i < nd && sub == 0) ro[i] = rc[i] - s;
      }
      collect(A.cres, res);
      scale(res);
      gemv32(true);
    }
  }

  __device__ void coarse(const Lev& L, VT* u) {
    __shared__ double rc[kTailDense], v[kTailDense], res[kTailDense];
    __shared__ float w[kTailDense];
    __shared__ double pow2[1];
    __shared__ unsigned red[32];
    static_assert(kTailThreads == 1024, "red holds one entry per warp");
    const int nd = A.nc * B;
    if (nd > 0) {
      if (nd <= kTailDenseBlock) coarse_dense<true>(L, rc, v, res, w, red, pow2, nd);
      else coarse_dense<false>(L, rc, v, res, w, red, pow2, nd);
    }
    for (int k = tid; k < L.n_r; k += nth) {
      const int c = __ldg(A.cidx + __ldg(A.gid + k));
#pragma unroll
      for (int b = 0; b < B; ++b)
        u[(size_t)b * L.n_r + k] = c >= 0 ? VT(v[c * B + b]) : VT(0);
    }
    sync();
  }

  // buffer that holds u of level k after `flips` updates
  static __device__ VT* buf(const Lev& L, int flips, int which) {
    return ((flips + which) & 1) ? L.u2 : L.u;
  }

  __device__ void run() {
    __shared__ VT wtab[kSupport];
    if (A.down) fill_weights(wtab);
    const int last = A.nlev - 1;
    const int per = A.smoother == RMG_SMOOTHER_GS ? 0
                  : A.smoother == RMG_SMOOTHER_JACOBI ? 1 : A.degree;
    if (A.down)
      for (int k = 0; k < last; ++k) {
        const Lev& L = A.lev[k];
        VT *cur = L.u, *oth = L.u2;
        smooth(L, cur, oth, A.nu1, true, false);
        sweep(L, cur, TailUpdate<OP_RESID_SCALED, VT>{L.r, L.b, nullptr, nullptr, nullptr, VT(0), VT(0)});
        restrict_to(L, A.lev[k + 1], wtab);
      }
    if (A.solve) coarse(A.lev[last], A.lev[last].u);
    if (A.up)
      for (int k = last - 1; k >= 0; --k) {
        const Lev& L = A.lev[k];
        const Lev& C = A.lev[k + 1];
        const VT* ubar = k + 1 == last ? C.u : buf(C, (A.nu1 + A.nu2) * per, 0);
        VT *cur = buf(L, A.nu1 * per, 0), *oth = buf(L, A.nu1 * per, 1);
        prolong(L, cur, C, ubar);
        smooth(L, cur, oth, A.nu2, false, true);
      }
  }
};

template <int DIM, int B, typename VT, typename CT>
__global__ void __launch_bounds__(kTailThreads, 1) k_tail(const __grid_constant__ TailArgs<VT, CT> A) {
  follow();
  // consecutive warps of the index go to different blocks, so that a level smaller than the
  // cluster uses all 16 SMs (the FP64 pipe of one SM takes 16 clocks for a warp's instruction)
  const int tid = (int)(((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31));
  Tail<DIM, B, VT, CT> t{A, tid, (int)(gridDim.x * blockDim.x)};
  t.run();
}


using KernelPtr = const void*;

template <typename VT, typename CT>
KernelPtr tail_kernel(int dim, int B) {
  if (dim == 3) return B == 1 ? (KernelPtr)k_tail<3, 1, VT, CT> : (KernelPtr)k_tail<3, 3, VT, CT>;
  return B == 1 ? (KernelPtr)k_tail<2, 1, VT, CT> : (KernelPtr)k_tail<2, 3, VT, CT>;
}

cudaLaunchConfig_t tail_config(int cluster, cudaLaunchAttribute* attr, cudaStream_t st) {
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = (unsigned)cluster;
  attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)cluster);
  cfg.blockDim = dim3(kTailThreads);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}
}  // namespace

void TailGeometry::build(Ctx& c, const Level& L, bool colours) {
  info.alloc(L.n_r);
  k_node_info<<<persistent_grid(c, (int)L.htiles.size()), kTile, 0, c.stream>>>(L.grid(),
                                                                               info.get());
  RMG_LAUNCHED();
  slots.alloc(std::max(1, L.nslots));
  if (L.nslots) {
    k_tail_slots<<<persistent_grid(c, (L.nslots + 255) / 256), 256, 0, c.stream>>>(
        L.nslots, L.sgrp.get(), L.gptr.get(), L.gslot.get(), slots.get());
    RMG_LAUNCHED();
  }
  if (!colours) return;
  std::vector<NodeInfo> in(L.n_r), out;
  RMG_CUDA(cudaMemcpyAsync(in.data(), info.get(), info.bytes(), cudaMemcpyDeviceToHost, c.stream));
  RMG_CUDA(cudaStreamSynchronize(c.stream));
  out.reserve(in.size());
  for (int k = 0; k < 8; ++k) {
    cstart[k] = (int)out.size();
    for (const NodeInfo& I : in)
      if (gs_colour_of<27>(I.ijl & 1023, (I.ijl >> 10) & 1023, I.ijl >> 20) == k) out.push_back(I);
  }
  cstart[8] = (int)out.size();
  coloured.alloc(out.size());
  RMG_CUDA(cudaMemcpy(coloured.get(), out.data(), coloured.bytes(), cudaMemcpyHostToDevice));
}

template <typename VT, typename CT>
int tail_cluster(int dim, int B) {
  const KernelPtr k = tail_kernel<VT, CT>(dim, B);
  auto allow_wide = [&] {            // an attribute of the function on the current device
    return cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
           cudaSuccess;
  };
  auto active = [&](int cluster, int* count) {
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = tail_config(cluster, &attr, nullptr);
    return cudaOccupancyMaxActiveClusters(count, k, &cfg) == cudaSuccess;
  };
  return widest_cluster(allow_wide, active, [] { cudaGetLastError(); });
}

template <typename VT, typename CT>
void tail_launch(int dim, int B, int cluster, bool next, const TailArgs<VT, CT>& args,
                 cudaStream_t st) {
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = tail_config(cluster, attr, st);
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // as launch_after
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.numAttrs = next ? 2 : 1;
  void* p[] = {const_cast<TailArgs<VT, CT>*>(&args)};
  RMG_CUDA(cudaLaunchKernelExC(&cfg, tail_kernel<VT, CT>(dim, B), p));
  RMG_LAUNCHED();
}

#define RMG_TAIL(VT, CT)                          \
  template int tail_cluster<VT, CT>(int, int);    \
  template void tail_launch<VT, CT>(int, int, int, bool, const TailArgs<VT, CT>&, cudaStream_t)
RMG_TAIL(double, double);
RMG_TAIL(float, float);
RMG_TAIL(float, __nv_bfloat16);
#undef RMG_TAIL

}  // namespace rmg
