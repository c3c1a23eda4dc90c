// Internal interface between the C-ABI host layer (es_host.cu) and the CUDA
// kernels (es_kernels.cu). Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "../../include/esopt.h"

namespace esopt {

// Elements per unit (what a thread takes at a time where a range is ragged)
// and per granule (what a launch divides between its CTAs; a segment takes a
// whole number of them, so a unit never spans two segments).
constexpr int kUnit = 8;
constexpr int kGranule = 16;
constexpr uint64_t granules_of(uint64_t numel) {
  return numel / kGranule + (numel % kGranule != 0 ? 1u : 0u);
}

// Threads per CTA of the diagnostic kernels (es_noise_bits, es_box_muller).
constexpr int kBlockThreads = 256;

// Bytes per element, per dtype.
constexpr size_t dtype_bytes(es_dtype_t dt) { return dt == ES_FP8_E4M3 ? 1u : dt == ES_BF16 ? 2u : 4u; }

// Device-side segment descriptor. A plan's table has nseg + 1 entries; the
// last is a sentinel whose granule_begin is the total number of granules.
struct SegDesc {
  void* data;              // 16-byte aligned storage of the segment
  uint64_t numel;          // elements in the segment
  uint64_t index_base;     // global index of element 0 (multiple of 8)
  uint64_t granule_begin;  // first granule of the segment in the plan's space
};
static_assert(sizeof(SegDesc) == 32, "SegDesc layout");

// A segment table small enough to travel as a launch parameter (2 KB).
constexpr int kTableSegments = 64;
struct SegTable {
  SegDesc entry[kTableSegments + 1];
};

// Largest number of generations one fused update launch applies.
constexpr int kMaxGenerations = 256;

// One fused update launch: `n_gen` generations of updates, generation g
// using seeds [gen_end[g-1], gen_end[g]) (gen_end[-1] = 0), each generation
// rounded to the storage type in turn; then, if `perturb`, one perturb step
// with (pkey, pscale). Passed by value as a kernel parameter (about 13 KB) and
// staged in shared memory by each CTA.
struct UpdateArgs {
  int n;          // seeds in all generations, 1..ES_MAX_SEEDS
  int n_gen;      // generations, 1..kMaxGenerations
  int perturb;    // 1: trailing perturb step
  float pscale;
  uint32_t pkey[2];
  uint16_t gen_end[kMaxGenerations];
  uint32_t key[ES_MAX_SEEDS][2];
  float coeff[ES_MAX_SEEDS];
};
static_assert(sizeof(UpdateArgs) < 32000, "kernel parameter limit");

struct PlanView {
  const SegDesc* segs;  // device table (nseg + 1 entries)
  int nseg;
  uint64_t granules;    // in all segments
  es_dtype_t dtype;
  // ES_FP8_E4M3: device array of 1 / scale per segment; NULL otherwise
  const float* inv_scale;
  // whether a launch may read the table before earlier work in its stream has
  // ended: true of a plan's own table, false of one that the stream itself copies
  bool early;
};

// Kernel launchers (es_kernels.cu). Each returns the launch's cudaError_t.
cudaError_t launch_axpy_noise(const PlanView& plan, uint64_t seed, float scale,
                              cudaStream_t stream);
// The same on bf16 or fp32 segments without a plan: nseg <= kTableSegments entries
// and the sentinel.
cudaError_t launch_axpy_table(const SegTable& table, int nseg, es_dtype_t dtype, uint64_t seed,
                              float scale, cudaStream_t stream);
cudaError_t launch_axpy_noise2(const PlanView& plan, uint64_t seed, float scale, uint64_t seed2,
                               float scale2, cudaStream_t stream);  // seed2 may equal seed
cudaError_t launch_update(const PlanView& plan, const UpdateArgs& args,
                          cudaStream_t stream);
cudaError_t launch_noise_bits(uint64_t seed, uint64_t block_base, uint64_t nblocks,
                              uint32_t* out, cudaStream_t stream);
cudaError_t launch_box_muller(const uint32_t* words, uint64_t npairs, float* out,
                              cudaStream_t stream);
cudaError_t launch_noise_fill(uint64_t seed, uint64_t index_base, uint64_t n,
                              float* out, cudaStream_t stream);

// Sets the calling thread's es_last_error() text (es_host.cu).
es_status_t record_status(es_status_t status, const char* message);

}  // namespace esopt
