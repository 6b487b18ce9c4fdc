// What sorted cells would leave out, estimated from a sample before anything is
// sorted, and the gates by which kernels that were launched for one route leave at
// once when the other one was taken.
#pragma once

#include "fms_internal.cuh"

namespace fms {

// How the cells' bounds are used: a seed against balls; against balls and extents
// (d > 8); a tile of seeds against tiles of points, out to weights of exactly zero.
enum ProbeKind : int { kProbeBall = 0, kProbeExtent = 1, kProbeTile = 2 };

// Of a seed's points, the share that the cells that it sees hold, up to which walking the
// cells pays: with every point visible a walk takes 1.2 to 1.6 times the dense kernels'
// time a pass, the first pass twice, after sorting (one update, d = 3 to 32: 2.4 to 3.4
// times in all; at shares of 0.02 to 0.2 0.1 to 0.5).  Clusters next to each other come
// out above 0.5, apart from each other below 0.3.
constexpr float kWalkShare = 0.35f;

constexpr int kProbeSets = 4;      // sets of a call that are sampled
constexpr int kProbePoints = 128;  // points and seeds of a sample
constexpr int kProbeSeeds = 16;

// Gated kernels follow each other in a chain of small launches.  On a stream they are
// launched while the one before still runs and wait for its end (and all that ended before
// it) themselves, which takes 1 us off each launch, empty or not.
__device__ __forceinline__ void wait_for_previous() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <typename... P, typename... A>
inline cudaError_t launch_gated(const Gate& gate, void (*kernel)(P...), dim3 grid, dim3 block,
                                size_t smem, cudaStream_t st, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = gate.chain ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

struct ProbeSet {
  const void* X;
  const void* Y;
  int64_t n, m;
};
struct ProbeArgs {
  ProbeSet set[kProbeSets];
  int sets, d, ld;   // rows of d values, ld apart
  double scale;
  int unit;          // 1: directions of the rows (cosine metric)
  int kind;
  float limit;       // share up to which *walk is 1
  float* share;      // [sets], device or mapped host memory
  int32_t* walk;     // [sets] or null
};
template <typename T>
cudaError_t launch_probe(const ProbeArgs& a, cudaStream_t st);

}  // namespace fms
