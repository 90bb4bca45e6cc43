// Launch helper shared by the translation units: phase A (region stencils, scalar or B x B
// blocks) and phase B (interface groups) with one epilogue.
#pragma once

#include <algorithm>
#include <cstdint>
#include <map>
#include <mutex>
#include <type_traits>
#include <unordered_map>
#include <utility>

#include "rmg_kernels.cuh"

namespace rmg {

// Blocks of kTile threads of `kernel` that one SM keeps resident (at most 8), queried once per
// kernel. A grid of more blocks than fit leaves its last ones to a second, sparse wave: sizing the
// grid of the 27-point half-plane sweeps by residency took a sweep of 10.6M nodes from 0.33 to
// 0.23 ms.
inline int resident_per_sm(const void* kernel) {
  static std::mutex m;
  static std::unordered_map<const void*, int> cache;
  std::lock_guard<std::mutex> lock(m);
  auto it = cache.find(kernel);
  if (it != cache.end()) return it->second;
  int b = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, kTile, 0) != cudaSuccess) {
    cudaGetLastError();
    b = 8;
  }
  b = std::max(1, std::min(b, 8));
  cache.emplace(kernel, b);
  return b;
}

// The same for a kernel with `smem` bytes of dynamic shared memory; also raises the kernel's
// dynamic shared memory limit, once per device (the attribute belongs to the device's context).
inline int resident_per_sm_smem(const void* kernel, int smem) {
  static std::mutex m;
  static std::map<std::pair<const void*, int>, int> cache;
  int dev = 0;
  RMG_CUDA(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lock(m);
  const auto key = std::make_pair(kernel, dev);
  auto it = cache.find(key);
  if (it != cache.end()) return it->second;
  int b = 0;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, kTile, smem) != cudaSuccess) {
    cudaGetLastError();
    b = 1;
  }
  b = std::max(1, std::min(b, 8));
  cache.emplace(key, b);
  return b;
}

// Whether the kernels of a level are launched with `next` below.
// In a graph, where the gaps between kernels are short already, up to 1.5M coefficients (a read of
// 12 MB in FP64, 3 to 6 us): next to longer kernels the waiting blocks are in the way. FP64 V-cycles
// with and without it on level 0, us: 672k nodes of 5 points (3.4M) 352 and 320, 1.33M of 7 (9.3M)
// 507 and 483, 256k of 27 (6.9M) 332 and 269.
// In a stream up to 40M: the power method of 3.1M nodes with 7 points gains 4 us a sweep, at 42M a
// solve with 7 points is level, at 970M one with 27 loses 4%.
inline bool short_kernels(const Level& L) {
  const long long coefs = (long long)L.n_r * L.kind * L.B * L.B;
  return coefs <= (g_capturing ? 1500000 : 40000000);
}
// The same for phase A of a product over run tiles in a stream. With long rows only up to 2M
// coefficients (two blocks an SM) and behind a phase B: the blocks are placed where those of the
// running kernel end first, and some SMs then get more of them than others. Products, us, phase A
// plain and dependent (phase B dependent in both): 27 points, 333k nodes 22.4 and 23.4, 817k 48.2
// and 51.5, 1.16M 65.9 and 69.8, 1.39M in uneven regions 76.9 and 86.5; one region of 54k without
// phase B 8.3 and 11.2; 7 points, 333k 10.4 and 8.8, 0.91M 18.5 and 16.7, 1.9M 34.9 and 33.1. Both
// plain and both dependent: 27 points, 74k nodes 12.4 and 8.7, 81k 12.4 and 15.5; blocks of 3 on 27
// points, 8k nodes (1.9M) 24.7 and 21.6, 22k 20.6 and 22.8, 169k 97 and 108.
inline bool short_product(const Level& L) {
  const int row = L.kind * L.B * L.B;
  return short_kernels(L) &&
         (g_capturing || row < 27 || (L.ngroups && (long long)L.n_r * row <= 2000000));
}

// kernel<<<grid, block, smem, st>>>(args...) for a kernel that starts with follow(). With `next`,
// where the work before it on the stream is a kernel too, it is set up while that one finishes
// (programmatic dependent launch), which takes about 1 us off each of the short kernels of a small
// problem; not beside an event record.
template <typename... P, typename... A>
void launch_after(bool next, void (*kernel)(P...), dim3 grid, int block, int smem,
                  cudaStream_t st, A&&... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = next ? 1 : 0;
  RMG_CUDA(cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...));
}
// launch_after with one resident wave of blocks over `work` tiles.
template <typename... P, typename... A>
void launch_resident(const Ctx& c, bool next, void (*kernel)(P...), int work, cudaStream_t st,
                     A&&... args) {
  const int g = persistent_grid(c, work, resident_per_sm((const void*)kernel));
  launch_after(next, kernel, dim3(g), kTile, 0, st, std::forward<A>(args)...);
}

// Phase B alone (scalar levels): one thread per copy of every interface group.
template <typename AT, class Epi>
void launch_groups(Ctx& c, const Level& L, const AT* y, Epi epi, cudaStream_t st,
                   bool next = true) {
  if (!L.ngroups) return;
  const int gs = persistent_grid(c, (L.nslots + 255) / 256);
  launch_after(next && short_kernels(L), k_groups<AT, Epi>, dim3(gs), 256, 0, st,
               L.nslots, L.slots.get(), L.gslot.get(), y, epi);
  RMG_LAUNCHED();
}

// The half-plane sweep of an FP32 level.
template <class Epi>
void launch_half(Ctx& c, const Level& L, const Grid& G, const float* coef, const float* half,
                 const int* asym, const float* u, float* y, Epi epi, cudaStream_t st, bool next) {
  const int nt = G.ntiles;
  const uint8_t* mu = L.mult.get();
  auto run = [&](auto kernel) {
    launch_resident(c, next, kernel, nt, st, G, coef, half, asym, u, mu, y, epi);
  };
  if (L.B == 3) {
    if (L.kind == 27) run(k_bstencil_half<27, 3, Epi>);
    else run(k_bstencil_half<9, 3, Epi>);
    return;
  }
  switch (L.kind) {
    case 5: run(k_stencil_half<5, Epi>); break;
    case 7: run(k_stencil_half<7, Epi>); break;
    case 9: run(k_stencil_half<9, Epi>); break;
    default: run(k_stencil_half<27, Epi>); break;
  }
}

// Phase A over `sweep` (a tuned tile list of L; the level's run tiles when null), then phase B.
// An FP32 sweep given half planes (see k_level0_fp32) and their asymmetry flag reads the half
// form while the flag is 0.
template <class Epi, typename CT, typename VT, typename AT>
void launch_stencil(Ctx& c, const Level& L, const CT* coef, const VT* u, AT* y, Epi epi,
                    cudaStream_t st, int* launches, cudaEvent_t ev0 = nullptr,
                    cudaEvent_t ev1 = nullptr, const Grid* sweep = nullptr,
                    const float* half = nullptr, const int* asym = nullptr) {
  Grid G = sweep ? *sweep : L.grid();
  // staged tiles copy 16-byte chunks: with an unaligned u or half-plane array the level's run
  // tiles take over
  if (G.lx == -3 && ((reinterpret_cast<uintptr_t>(u) | reinterpret_cast<uintptr_t>(half)) & 15))
    G = L.grid();
  const int gb = persistent_grid(c, G.ntiles);
  const bool next = !ev0 && (sweep ? short_kernels(L) : short_product(L));
  // external record nodes when capturing, so the events can be timed after a graph replay
  if (ev0) RMG_CUDA(cudaEventRecordWithFlags(ev0, st, g_capturing ? cudaEventRecordExternal : 0));
  bool done = false;
  if constexpr (std::is_same<CT, float>::value && std::is_same<VT, float>::value &&
                std::is_same<AT, float>::value) {
    if (half && L.B == 1 && G.lx == -3) {
      RMG_REQUIRE(asym != nullptr && L.kind == 27, RMG_ERR_STATE,
                  "staged sweeps need the half planes of a 27-point stencil");
      const int smem = kStSmemFloats * (int)sizeof(float);
      const auto kern = k_stencil_half27_staged<Epi>;
      const int g = persistent_grid(c, G.ntiles, resident_per_sm_smem((const void*)kern, smem));
      launch_after(next, kern, dim3(g), kStX * kStY, smem, st, G, coef, half, asym, u,
                   L.mult.get(), y, epi);
      done = true;
    } else if (half && L.B == 1) {
      RMG_REQUIRE(asym != nullptr, RMG_ERR_STATE, "half planes without their flag");
      launch_half(c, L, G, coef, half, asym, u, y, epi, st, next);
      done = true;
    } else if (half) {
      RMG_REQUIRE(asym != nullptr && L.B == 3 && (L.kind == 27 || L.kind == 9), RMG_ERR_STATE,
                  "half planes of a block operator need 3 dofs and a 27- or 9-point stencil");
      launch_half(c, L, G, coef, half, asym, u, y, epi, st, next);
      done = true;
    }
  }
  RMG_REQUIRE(done || G.lx != -3, RMG_ERR_STATE, "staged tiles outside a half-plane sweep");
  auto run = [&](auto kernel) {
    launch_after(next, kernel, dim3(gb), kTile, 0, st, G, coef, u, L.mult.get(), y, epi);
  };
  if (done) {
  } else if (L.B == 1) {
    switch (L.kind) {
      case 5: run(k_stencil<5, CT, VT, AT, Epi>); break;
      case 7: run(k_stencil<7, CT, VT, AT, Epi>); break;
      case 9: run(k_stencil<9, CT, VT, AT, Epi>); break;
      default: run(k_stencil<27, CT, VT, AT, Epi>); break;
    }
  } else {
    RMG_REQUIRE(L.B == 3 && (L.kind == 27 || L.kind == 9), RMG_ERR_ARG,
                "block operators need 3 dofs per node and a 27- or 9-point stencil");
    if (L.kind == 27)
      run(k_bstencil<27, 3, CT, VT, AT, Epi>);
    else
      run(k_bstencil<9, 3, CT, VT, AT, Epi>);
  }
  RMG_LAUNCHED();
  if (ev1) RMG_CUDA(cudaEventRecordWithFlags(ev1, st, g_capturing ? cudaEventRecordExternal : 0));
  if (launches) ++*launches;
  if (L.ngroups) {
    if (L.B == 1) {
      launch_groups(c, L, y, epi, st, !ev1);
    } else {
      const int gg = persistent_grid(c, (L.nslots + 255) / 256);
      launch_after(!ev1 && short_kernels(L), k_groups_b<AT, Epi>, dim3(gg), 256, 0, st,
                   L.nslots, L.B, L.n_r, L.slots.get(), L.gslot.get(), (const AT*)y, epi);
      RMG_LAUNCHED();
    }
    if (launches) ++*launches;
  }
}

}  // namespace rmg
