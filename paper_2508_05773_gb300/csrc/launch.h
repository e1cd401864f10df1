// launch.h -- host-side interface between the C ABI and the solve kernels.
#pragma once

#include <cuda_runtime.h>

#include "rollout.cuh"

namespace brmppi {

using KernelFn = void (*)(const KConst, const LaunchDesc);

struct Variant {
  int tps, bpt;
  int family;  // Family
  KernelFn fn;
  int rows = 0;  // > 0: exactly this many constraint rows a lane (single solves)
  int ns = 1;    // samples a team rolls out together
  bool local = false;  // rows' state in local memory
};

// Instantiations (variants.h): each function returns its table and its length.
const Variant* variants_narrow_plain(int* n);
const Variant* variants_narrow_discs(int* n);
const Variant* variants_narrow_point(int* n);
const Variant* variants_narrow_moving(int* n);
const Variant* variants_wide_plain(int* n);
const Variant* variants_wide_discs(int* n);
const Variant* variants_wide_point(int* n);
const Variant* variants_wide_moving(int* n);
const Variant* variants_latency_plain(int* n);
const Variant* variants_latency_discs(int* n);
const Variant* variants_latency_point(int* n);
const Variant* variants_latency_moving(int* n);

// The family a launch with these constants takes.
inline int family_of(const KConst& k) {
  if (k.discs) return kDiscs;
  if (k.third || k.jerk || k.abuf) return kPoint;
  return k.obs8 || k.coll ? kMoving : kPlain;
}

// Threads of a launch shape.  `threads` / tps is the samples of a CTA's tile;
// with ns samples a team threads / ns of them roll out.  Teams of one sample
// wider than one lane with at most two Philox blocks per lane add warps that
// produce the noise, enough for two blocks per producer lane and step where
// the CTA has room (up to four; P blocks per sample).  Other variants draw on
// their own lanes (0 noise warps).  At most kMaxBlockThreads (the kernels'
// launch bound).
constexpr int kMaxBlockThreads = 512;
constexpr int kMaxRowsBlockThreads = 384;  // the exact-rows instantiations' launch bound
// How a shape is run: samples a team, and the rows' state in local memory
// (where it does not fit in shared memory; one sample a team).
struct LaunchMode {
  int ns = 1;
  bool local = false;
};
int noise_warps(int tps, int bpt, int threads, int P, int ns = 1);
int block_threads(int tps, int bpt, int threads, int P, int ns = 1);

// The rows a lane holds in a single solve of n_rows constraint rows on a
// noise-warp shape, if the instantiation with exactly that many is compiled
// (LaunchDesc::rows), else 0.
int exact_rows_variant(int tps, int bpt, const KConst& k, int n_rows);

// Supported (threads per sample, Philox blocks per lane) pairs.
bool variant_exists(int tps, int bpt);
// Whether a pair is compiled with two samples a team.
bool pair_exists(int tps, int bpt, int family);

// Raise the dynamic shared-memory limit of every variant to `bytes`.
cudaError_t set_smem_limit(size_t bytes);

// CTAs of a variant resident per SM for a launch shape (0 if it cannot run).
int variant_occupancy(int tps, int bpt, int threads, size_t smem, int family, int P, LaunchMode mode);

// Enqueue the hitch stabilizer for n states (out: n x 4 floats).
cudaError_t launch_stabilize(const KConst& k, const double* x, const float* u_ref, int n, float* out,
                             cudaStream_t stream);

// Enqueue the hitch stabilizer for the instances of a device table whose
// u_safe is set (after their solve, on the same stream).
cudaError_t launch_stabilize_table(const KConst& k, const Inst* d_table, int n, cudaStream_t stream);

// Enqueue the noise-table kernel: Philox words and Box-Muller normals of
// samples < n_samples, steps < H, blocks < n_blocks (words or normals may
// be null).
cudaError_t launch_noise_blocks(uint64_t seed, uint64_t counter, int n_samples, int H, int n_blocks, uint32_t* words,
                                float* normals, cudaStream_t stream);

// Enqueue the one-CTA merge of an instance's gathered tile partials
// (in.part, in.tiles; caps: the instance's tables; smem: their bytes).
cudaError_t launch_merge_tiles(const KConst& k, const Inst& in, const SmemCaps& caps, size_t smem,
                               cudaStream_t stream);

// Enqueue one launch of the solve kernel.
cudaError_t launch_solve(int tps, int bpt, int blocks, int threads, size_t smem, cudaStream_t stream,
                         const KConst& k, const LaunchDesc& L, int P, LaunchMode mode);

}  // namespace brmppi
