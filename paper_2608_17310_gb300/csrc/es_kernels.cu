// sm_103a kernels of the ES step: in-place perturb/restore (theta += s eps) and
// the fused N-seed update (theta += sum_i c_i eps_i), plus a noise fill.
//
// Both stream the parameter set once per launch. A plan's segments lie end to
// end in a space of 16-element granules; a launch cuts that space into one
// contiguous range per CTA, all of one length, with one large CTA per SM. A CTA
// finds its first segment by a search and walks its range from there, so every
// SM gets the same work whatever the set's size and however it is divided into
// tensors.
// Every element is owned by exactly one thread: no atomics, no shared state
// between threads except the staged seeds of the update and, on small sets, the
// polar forms that its warps hand over.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>

#include "es_internal.h"
#include "es_noise.cuh"

namespace esopt {
namespace {

// Stored vector <-> fp32 registers, and units of 8 elements, whole or cut off.
struct Bf16Io {
  static constexpr int kVec = 8;
  static constexpr bool kScaled = false;
  using Scalar = uint16_t;
  using Vec = uint4;  // what a thread loads at once in a run
  using Raw = uint4;  // a unit of 8 elements as stored
  __device__ static uint32_t pack2(float lo, float hi) {
    __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);  // one cvt.rn.bf16x2.f32
    return *reinterpret_cast<uint32_t*>(&h);
  }
  __device__ static float lo(uint32_t w) { return __uint_as_float(w << 16); }
  __device__ static float hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }
  __device__ static void unpack(const uint4& v, float (&f)[8]) {
    f[0] = lo(v.x); f[1] = hi(v.x);
    f[2] = lo(v.y); f[3] = hi(v.y);
    f[4] = lo(v.z); f[5] = hi(v.z);
    f[6] = lo(v.w); f[7] = hi(v.w);
  }
  __device__ static uint4 pack(const float (&f)[8]) {
    return make_uint4(pack2(f[0], f[1]), pack2(f[2], f[3]), pack2(f[4], f[5]), pack2(f[6], f[7]));
  }
  // f <- value of round_to_storage(f), element-wise (one rounding to bf16). kSingly:
  // with 0 in the low half the converted pair is the rounded value's fp32 bits, one
  // instruction an element, where packing two and unpacking them takes three for
  // both: the flip 621 -> 612 us over 792,680,960 parameters. The two-step pass,
  // which has no register to spare, is faster through the pairs (1093 against 1099).
  template <bool kSingly, int M>
  __device__ static void round_trip(float (&f)[M]) {
#pragma unroll
    for (int k = 0; k < M; k += 2) {
      if constexpr (kSingly) {
        f[k] = __uint_as_float(pack2(0.0f, f[k]));
        f[k + 1] = __uint_as_float(pack2(0.0f, f[k + 1]));
      } else {
        const uint32_t w = pack2(f[k], f[k + 1]);
        f[k] = lo(w);
        f[k + 1] = hi(w);
      }
    }
  }
  // The first `rem` (1 .. 8) elements of the unit at p, the rest zero.
  __device__ static Raw load_unit(const uint16_t* p, int rem) {
    if (rem == kUnit) return *reinterpret_cast<const uint4*>(p);
    uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int k = 0; k < kUnit; ++k)
      if (k < rem) w[k >> 1] |= static_cast<uint32_t>(p[k]) << (16 * (k & 1));
    return make_uint4(w[0], w[1], w[2], w[3]);
  }
  __device__ static void store_unit(uint16_t* p, int rem, const Raw& v) {
    if (rem == kUnit) {
      *reinterpret_cast<uint4*>(p) = v;
      return;
    }
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int k = 0; k < kUnit; ++k)
      if (k < rem) p[k] = static_cast<uint16_t>(w[k >> 1] >> (16 * (k & 1)));
  }
  __device__ static Raw zero_unit() { return make_uint4(0u, 0u, 0u, 0u); }
  // one element: its value, the stored form of a value, and that form's value
  __device__ static float value(uint16_t h) { return __uint_as_float(static_cast<uint32_t>(h) << 16); }
  __device__ static uint16_t store(float f) { return static_cast<uint16_t>(pack2(f, 0.0f)); }
  __device__ static void unpack_unit(const Raw& v, float (&f)[kUnit]) { unpack(v, f); }
  __device__ static Raw pack_unit(const float (&f)[kUnit]) { return pack(f); }
};

struct F32Io {
  static constexpr int kVec = 4;
  static constexpr bool kScaled = false;
  using Scalar = float;
  using Vec = uint4;
  __device__ static void unpack(const uint4& v, float (&f)[4]) {
    f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y);
    f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
  }
  __device__ static uint4 pack(const float (&f)[4]) {
    return make_uint4(__float_as_uint(f[0]), __float_as_uint(f[1]),
                      __float_as_uint(f[2]), __float_as_uint(f[3]));
  }
  template <bool, int M>
  __device__ static void round_trip(float (&)[M]) {}
  struct Raw {
    uint4 lo, hi;
  };
  __device__ static float value(float f) { return f; }
  __device__ static float store(float f) { return f; }
  __device__ static Raw load_unit(const float* p, int rem) {
    if (rem == kUnit) {
      const uint4* q = reinterpret_cast<const uint4*>(p);
      return Raw{q[0], q[1]};
    }
    float f[kUnit];
#pragma unroll
    for (int k = 0; k < kUnit; ++k) f[k] = k < rem ? p[k] : 0.0f;
    return pack_unit(f);
  }
  __device__ static void store_unit(float* p, int rem, const Raw& v) {
    if (rem == kUnit) {
      uint4* q = reinterpret_cast<uint4*>(p);
      q[0] = v.lo;
      q[1] = v.hi;
      return;
    }
    float f[kUnit];
    unpack_unit(v, f);
#pragma unroll
    for (int k = 0; k < kUnit; ++k)
      if (k < rem) p[k] = f[k];
  }
  __device__ static Raw zero_unit() {
    return Raw{make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
  }
  __device__ static void unpack_unit(const Raw& v, float (&f)[kUnit]) {
    const uint32_t w[kUnit] = {v.lo.x, v.lo.y, v.lo.z, v.lo.w, v.hi.x, v.hi.y, v.hi.z, v.hi.w};
#pragma unroll
    for (int k = 0; k < kUnit; ++k) f[k] = __uint_as_float(w[k]);
  }
  __device__ static Raw pack_unit(const float (&f)[kUnit]) {
    return Raw{make_uint4(__float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]),
                          __float_as_uint(f[3])),
               make_uint4(__float_as_uint(f[4]), __float_as_uint(f[5]), __float_as_uint(f[6]),
                          __float_as_uint(f[7]))};
  }
};

// FP8 E4M3 storage: 8 elements per 8-byte vector, byte k of the vector is
// element k. Values stay in units of the segment's scale: the kernels multiply
// the noise by 1 / scale instead (kScaled). Decoding goes through half
// precision, which holds every E4M3 value exactly; encoding rounds fp32 to the
// nearest E4M3 value, ties to even, saturating at +-448 (cvt .satfinite).
struct Fp8Io {
  static constexpr int kVec = 8;
  static constexpr bool kScaled = true;
  using Scalar = uint8_t;
  using Vec = uint2;
  using Raw = uint2;
  __device__ static float2 dec2(uint32_t pair) {
    const __half2_raw h =
        __nv_cvt_fp8x2_to_halfraw2(static_cast<__nv_fp8x2_storage_t>(pair & 0xFFFFu), __NV_E4M3);
    return __half22float2(__half2(h));
  }
  __device__ static uint32_t enc2(float lo, float hi) {
    return static_cast<uint32_t>(__nv_cvt_float2_to_fp8x2(make_float2(lo, hi), __NV_SATFINITE,
                                                          __NV_E4M3));
  }
  __device__ static void unpack(const uint2& v, float (&f)[8]) {
    const uint32_t w[2] = {v.x, v.y};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float2 a = dec2(w[k]), b = dec2(w[k] >> 16);
      f[4 * k + 0] = a.x; f[4 * k + 1] = a.y; f[4 * k + 2] = b.x; f[4 * k + 3] = b.y;
    }
  }
  __device__ static uint2 pack(const float (&f)[8]) {
    return make_uint2(enc2(f[0], f[1]) | (enc2(f[2], f[3]) << 16),
                      enc2(f[4], f[5]) | (enc2(f[6], f[7]) << 16));
  }
  template <bool, int M>
  __device__ static void round_trip(float (&f)[M]) {
#pragma unroll
    for (int k = 0; k < M; k += 2) {
      const float2 r = dec2(enc2(f[k], f[k + 1]));
      f[k] = r.x;
      f[k + 1] = r.y;
    }
  }
  __device__ static float value(uint8_t c) { return dec2(c).x; }
  __device__ static uint8_t store(float f) { return static_cast<uint8_t>(enc2(f, 0.0f)); }
  __device__ static Raw load_unit(const uint8_t* p, int rem) {
    if (rem == kUnit) return *reinterpret_cast<const uint2*>(p);
    uint32_t w[2] = {0u, 0u};
#pragma unroll
    for (int k = 0; k < kUnit; ++k)
      if (k < rem) w[k >> 2] |= static_cast<uint32_t>(p[k]) << (8 * (k & 3));
    return make_uint2(w[0], w[1]);
  }
  __device__ static void store_unit(uint8_t* p, int rem, const Raw& v) {
    if (rem == kUnit) {
      *reinterpret_cast<uint2*>(p) = v;
      return;
    }
    const uint32_t w[2] = {v.x, v.y};
#pragma unroll
    for (int k = 0; k < kUnit; ++k)
      if (k < rem) p[k] = static_cast<uint8_t>(w[k >> 2] >> (8 * (k & 3)));
  }
  __device__ static Raw zero_unit() { return make_uint2(0u, 0u); }
  __device__ static void unpack_unit(const Raw& v, float (&f)[kUnit]) { unpack(v, f); }
  __device__ static Raw pack_unit(const float (&f)[kUnit]) { return pack(f); }
};

// theta + acc in storage units: acc is in parameter units, so a scaled
// segment takes acc / scale (one fused multiply-add with 1 / scale).
template <class Io>
__device__ __forceinline__ float add_acc(float theta, float acc, float inv_scale) {
  if constexpr (Io::kScaled) return fmaf(acc, inv_scale, theta);
  else return theta + acc;
}

// Philox words of one seed's blocks that share the high counter word, with the
// round keys read from a precomputed schedule (kernel parameters, or registers
// loaded from shared memory) and the constants of that word given.
template <class Keys, bool kWideFirst = false>
struct SchedGen {
  TileConst t;
  uint32_t rk1, rk2;  // round 0's k1, round 1's k0
  Keys rk;            // rounds 2..9: rk[2r - 4], rk[2r - 3]
  // From round 0's product (philox_round0 of the block's low counter word).
  __device__ uint4 block_r0(Round0 p0) const {
    return philox_block_r0<kWideFirst>(p0, t, rk1, rk2, rk);
  }
};

// Generator of one seed whose schedule is a kernel parameter.
template <bool kWideFirst>
__device__ __forceinline__ SchedGen<const uint32_t*, kWideFirst> sched_gen(const PhiloxSched& s,
                                                                          uint32_t j_hi) {
  return {tile_const(j_hi, s.rk[0], s.rk[3]), s.rk[1], s.rk[2], s.rk + 4};
}

// The pairs of NB Philox blocks in polar form (r, cos, sin) from their words,
// with packed two-wide FP32 instructions (each half rounds exactly like the
// scalar instruction) and the near-one radius inputs on a rare branch.
template <int NB>
__device__ __forceinline__ void polar_from_words(const uint4 (&x)[NB], Polar2 (&p)[NB]) {
  uint2 xa[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    xa[b] = make_uint2(x[b].x, x[b].z);
    p[b] = polar2_sq(x[b]);
  }
  fix_near_one<NB>(xa, p);
#pragma unroll
  for (int b = 0; b < NB; ++b) p[b].r = make_float2(sqrt_approx(p[b].r.x), sqrt_approx(p[b].r.y));
}

// f[k] += scale * eps[4 j0 + k] for the V elements of blocks whose polar
// forms are pp, with scale folded into each pair's radius.
template <int V>
__device__ __forceinline__ void apply_noise(const Polar2 (&pp)[V / 4], float scale, float (&f)[V]) {
#pragma unroll
  for (int b = 0; b < V / 4; ++b) {
    const Polar2& p = pp[b];
    const float2 sr = __fmul2_rn(make_float2(-scale, -scale), p.r);   // -(scale * r)
    const float2 lo = __ffma2_rn(make_float2(sr.x, sr.x), make_float2(p.c.x, p.s.x),
                                 make_float2(f[4 * b + 0], f[4 * b + 1]));
    const float2 hi = __ffma2_rn(make_float2(sr.y, sr.y), make_float2(p.c.y, p.s.y),
                                 make_float2(f[4 * b + 2], f[4 * b + 3]));
    f[4 * b + 0] = lo.x;
    f[4 * b + 1] = lo.y;
    f[4 * b + 2] = hi.x;
    f[4 * b + 3] = hi.y;
  }
}

// f[k] += scale * eps for the V elements of the Philox blocks whose words
// are x.
template <int V>
__device__ __forceinline__ void add_scaled_noise(const uint4 (&x)[V / 4], float scale,
                                                 float (&f)[V]) {
  Polar2 pp[V / 4];
  polar_from_words<V / 4>(x, pp);
  apply_noise<V>(pp, scale, f);
}

// Segment of `granule`, at or after `lo` (segs[lo].granule_begin <= granule):
// the warp tests 32 evenly spaced entries at a time, one per lane, so a table
// of n segments takes log32(n) dependent loads. The loads are L2 latency and
// nothing else: on a set of 200 ragged tensors a walk from entry 0 was most of a
// launch (40 us of which a search leaves 5). Called by whole warps; every lane
// returns the same segment.
__device__ __forceinline__ int search_segment(const SegDesc* __restrict__ segs, int lo, int nseg,
                                              uint64_t granule) {
  const int lane = static_cast<int>(threadIdx.x & 31u);
  int hi = nseg;  // granule < segs[hi].granule_begin
  while (hi - lo > 1) {
    const int step = (hi - lo + 31) / 32;
    const int probe = lo + step * (lane + 1);
    const bool passed = probe < hi && segs[probe].granule_begin <= granule;
    const int c = __popc(__ballot_sync(0xFFFFFFFFu, passed));  // a prefix of the lanes
    lo += step * c;
    hi = lo + step < hi ? lo + step : hi;
  }
  return lo;
}

// The same among segments lo .. hi by one thread alone (bisection).
__device__ __forceinline__ int segment_between(const SegDesc* __restrict__ segs, int lo, int hi,
                                               uint64_t granule) {
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (segs[mid].granule_begin <= granule) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Programmatic dependent launch: a kernel lets the next one in its stream start
// when its own CTAs are done, and waits, before it touches the parameters, until
// the one before it has completed with its writes visible. What runs ahead is the
// launch itself, 2-3 us in a stream, and the segment search: passes over 2^20
// parameters in a stream 6.2 -> 3.3 us each, over 2^24 18.5 -> 15.9. Letting the next
// one start at a kernel's beginning gained nothing more, and on small grids packed
// its waiting CTAs onto few SMs (128 seeds over 65,536 parameters 22.8 -> 27.4 us).
__device__ __forceinline__ void let_next_start() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void wait_for_previous() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// A launch's division of the plan: `granules` in ranges of `per_cta`, the last
// one shorter. The host makes the grid so that no range is empty.
struct Split {
  uint64_t granules;
  uint64_t per_cta;
};
constexpr int kUnitsPerGranule = kGranule / kUnit;

__device__ __forceinline__ uint64_t range_begin(const Split& s) { return blockIdx.x * s.per_cta; }
__device__ __forceinline__ uint64_t range_end(const Split& s) {
  const uint64_t e = range_begin(s) + s.per_cta;
  return e < s.granules ? e : s.granules;
}

// The unit of 8 elements that a thread takes from a range: `rem` of them lie in
// the segment (0: none).
template <class Io>
struct UnitRef {
  typename Io::Scalar* p;
  int rem;
  uint64_t j0;  // Philox block of element 0 (index bases are multiples of 8)
  float inv;    // 1 / the segment's scale, for a scaled storage type
};

template <class Io>
__device__ __forceinline__ UnitRef<Io> unit_ref(const SegDesc& d, float inv,
                                                uint64_t unit) {
  const uint64_t e = (unit - d.granule_begin * kUnitsPerGranule) * kUnit;
  UnitRef<Io> r;
  r.rem = e >= d.numel ? 0 : d.numel - e < kUnit ? static_cast<int>(d.numel - e) : kUnit;
  r.p = static_cast<typename Io::Scalar*>(d.data) + e;
  r.j0 = (d.index_base + e) >> 2;
  r.inv = inv;
  return r;
}

// What a pass over the parameters does: one step theta += scale1 * eps_seed1;
// two steps, the second on the first's result rounded to the storage type
// (restore of one member fused with the perturb of the next); the two steps
// of one seed, whose noise is generated once (the antithetic flip); or the update
// of a population of 1 to 8, theta += sum_i scale_i eps_seed_i rounded once, which
// the next generation's first perturb may follow on the rounded result.
enum class AxpyKind { kSteps, kFlip, kSum, kSumPerturb };
constexpr int kMaxSum = 8;

// What a pass does, and the number of its seeds' schedules (kSumPerturb: the last
// one is the perturb's).
template <AxpyKind kKind, int kSeedCount>
struct AxpyMode {
  static constexpr AxpyKind kind = kKind;
  static constexpr int seeds = kSeedCount;
  static constexpr bool sum = kKind == AxpyKind::kSum || kKind == AxpyKind::kSumPerturb;
};
using AxpyOne = AxpyMode<AxpyKind::kSteps, 1>;
using AxpyTwo = AxpyMode<AxpyKind::kSteps, 2>;
using AxpyFlip = AxpyMode<AxpyKind::kFlip, 1>;
template <int N>
using AxpySum = AxpyMode<AxpyKind::kSum, N>;
template <int N>
using AxpySumPerturb = AxpyMode<AxpyKind::kSumPerturb, N + 1>;

// Arguments of a launch: each seed's schedule, and the scale of each step or
// seed. A __grid_constant__ parameter, so every round key is read from the
// constant bank as an instruction operand.
struct AxpyArgs {
  PhiloxSched seed[kMaxSum + 1];
  float scale[kMaxSum + 1];
};

// The steps of Mode on the V values f. words(i, x) gives the Philox words of
// seed i's blocks; inv is 1 / the segment's scale.
template <class Io, class Mode, int V, class Words>
__device__ __forceinline__ void axpy_values(const Words& words, const AxpyArgs& a, float inv,
                                            float (&f)[V]) {
  constexpr int kSeeds = Mode::seeds;
  uint4 x[V / 4];
  words(0, x);
  if constexpr (Mode::sum) {
    float acc[V];
#pragma unroll
    for (int k = 0; k < V; ++k) acc[k] = 0.0f;
    // each seed's words before the transform of the one before (2 % faster than
    // after it; the two-step pass does not gain from it)
    constexpr bool kPerturb = Mode::kind == AxpyKind::kSumPerturb;
    constexpr int kSummed = kSeeds - (kPerturb ? 1 : 0);
#pragma unroll
    for (int i = 0; i < kSummed; ++i) {
      uint4 y[V / 4];
      if (i + 1 < kSeeds) words(i + 1, y);
      add_scaled_noise<V>(x, a.scale[i], acc);
      if (i + 1 < kSeeds) {
#pragma unroll
        for (int b = 0; b < V / 4; ++b) x[b] = y[b];
      }
    }
#pragma unroll
    for (int k = 0; k < V; ++k) f[k] = add_acc<Io>(f[k], acc[k], inv);
    if constexpr (kPerturb) {
      Io::template round_trip<true>(f);
      add_scaled_noise<V>(x, a.scale[kSummed] * inv, f);
    }
  } else if constexpr (Mode::kind == AxpyKind::kFlip) {
    Polar2 pp[V / 4];
    polar_from_words<V / 4>(x, pp);
    apply_noise<V>(pp, a.scale[0] * inv, f);
    Io::template round_trip<true>(f);
    apply_noise<V>(pp, a.scale[1] * inv, f);
  } else {
    add_scaled_noise<V>(x, a.scale[0] * inv, f);
    if constexpr (kSeeds == 2) {
      Io::template round_trip<false>(f);
      words(1, x);
      add_scaled_noise<V>(x, a.scale[1] * inv, f);
    }
  }
}

// The generators of a launch's seeds for one high counter word.
template <class Mode, bool kWide>
struct AxpyGens {
  static constexpr int kSeeds = Mode::seeds;
  TileConst t[kSeeds];
  __device__ AxpyGens(const AxpyArgs& a, uint32_t j_hi) {
#pragma unroll
    for (int i = 0; i < kSeeds; ++i) t[i] = tile_const(j_hi, a.seed[i].rk[0], a.seed[i].rk[3]);
  }
  __device__ uint4 words(const AxpyArgs& a, int i, Round0 p0) const {
    const uint32_t* rk = a.seed[i].rk;
    return philox_block_r0<kWide>(p0, t[i], rk[1], rk[2], rk + 4);
  }
};

// Shape of a pass: threads of its one CTA per SM, vectors per thread in a tile
// (the unrolled body of the loop) and how many vectors ahead theta is loaded. What
// bounds the passes is the generator's instruction stream: the FMA-heavy pipe
// (integer products), MUFU and issue. All of an SM's warps in one CTA on a short
// loop body run 6-15 % faster than 2 or 3 CTAs of 256 threads on a body of four
// vectors. Measured on sm_103a over 792,680,960 parameters (us; 256 threads, 4
// vectors, 1 ahead, grid-stride tiles -> this): bf16 one step 678 -> 569 (5.58 TB/s),
// two steps 1217 -> 1093 (1.450e12 Gaussians/s), flip 729 -> 612; fp32 971 -> 960 (6.6
// TB/s: HBM), 1366 -> 1077, 976 -> 961; FP8 636 -> 570, 1301 -> 1118, 718 -> 635 (8
// elements at a time: 16 hold twice the registers and body, and cost the sums of 4 and
// more seeds 1-10 %).
// The sums replace the seed loop of update_kernel, which spends a third of a seed
// per unit filling and draining its pipeline and reads each seed's keys from shared
// memory: 1 / 2 / 3 / 4 / 8 seeds bf16 972 / 1480 / 2035 / 2555 / 4700 -> 591 / 1075 /
// 1604 / 2107 / 4183 (the seed loop as it is now: 4404 at 8), fp32 1125 / 1642 / 2253 /
// 2866 / 5314 -> 962 / 1088 / 1589 / 2145 / 4351, FP8 811 / 1392 / 1979 / 2567 / 4902 -> 589 /
// 1088 / 1579 / 2115 / 4171; with the perturb behind 1 / 4 / 8 bf16 seeds 1656 / 3249 / 5433
// -> 1107 / 2675 / 4752. 12 and 16 seeds unrolled gain 3 and 1 % on the loop, for twice
// the code: not built.
// fp32: 4 vectors, 2 ahead, while HBM bounds the pass (perturb 958, against 1133 with
// one vector) and as far as that body fits into 64 registers with few spills (4
// schedules 2167 against 2182, with 220 bytes spilled; 896 threads 2161, 768 2213); from
// 5 on one vector (5 schedules 2858 -> 2745, 8 6243 -> 4354).
// Thread counts that are no multiple of 128 leave the SM's four schedulers
// unequal warps and run 10 % slower.
struct AxpyShape {
  int threads, vecs, ahead;
};
template <class Io, class Mode>
__host__ __device__ constexpr AxpyShape axpy_shape() {
  if (Io::kVec == 4) return Mode::seeds > 4 ? AxpyShape{1024, 1, 1} : AxpyShape{1024, 4, 2};
  if (Mode::sum)
    return Mode::seeds == 1 || (Mode::seeds == 2 && !Io::kScaled) ? AxpyShape{1024, 2, 2}
           : Mode::seeds <= 3                                     ? AxpyShape{896, 2, 2}
           : Mode::seeds <= 7                                     ? AxpyShape{768, 1, 1}
                                                                  : AxpyShape{640, 1, 1};
  if (Mode::kind == AxpyKind::kFlip) return {1024, 3, 1};
  if (Mode::seeds == 1) return {1024, 2, 2};
  return Io::kScaled ? AxpyShape{768, 2, 2} : AxpyShape{1024, 2, 1};
}
// Units of one tile.
template <class Io, class Mode>
__host__ __device__ constexpr uint64_t axpy_tile_units() {
  constexpr AxpyShape k = axpy_shape<Io, Mode>();
  return static_cast<uint64_t>(k.threads) * k.vecs * Io::kVec / kUnit;
}

// `tiles` whole tiles of one segment, all with the same high counter word,
// from the calling thread's first vector at p, whose first Philox block is
// j_thread. Vector u of a tile is one 16-byte vector per thread (FP8: 8 bytes), so
// each load and store instruction of a warp covers 512 (256) contiguous bytes; the load of the
// vector `ahead` of the current one is issued before that is computed. Round 0's Philox
// product (of the counter alone) is stepped by 64-bit additions from the
// thread's first block instead of multiplied.
template <class Io, class Mode>
__device__ __forceinline__ void axpy_run(typename Io::Scalar* p, uint64_t j_thread, uint32_t tiles,
                                         const AxpyArgs& a, float inv) {
  constexpr int V = Io::kVec, NB = V / 4;
  constexpr AxpyShape kShape = axpy_shape<Io, Mode>();
  constexpr int D = kShape.ahead;
  constexpr int kStride = kShape.threads * V;  // elements between a thread's vectors
  static_assert(kShape.vecs % D == 0, "the vectors in flight rotate within a tile");
  // the one-seed pass is fastest with every Philox product 64-bit wide (FP8, the
  // least of the three: 572.7 -> 570.6 us over 792,680,960 parameters)
  constexpr bool kWide = Mode::kind == AxpyKind::kSteps && Mode::seeds == 1;
  const uint32_t j_hi = static_cast<uint32_t>(j_thread >> 32);
  const AxpyGens<Mode, kWide> gens(a, j_hi);
  Round0 p0 = philox_round0<kWide>(static_cast<uint32_t>(j_thread));
  typename Io::Vec v[D];
#pragma unroll
  for (int k = 0; k < D; ++k) v[k] = *reinterpret_cast<const typename Io::Vec*>(p + k * kStride);
#pragma unroll 1
  for (;;) {
#pragma unroll
    for (int u = 0; u < kShape.vecs; ++u) {
      float f[V];
      Io::unpack(v[u % D], f);
      if (u + D < kShape.vecs || tiles > 1)
        v[u % D] = *reinterpret_cast<const typename Io::Vec*>(p + (u + D) * kStride);
      Round0 r0[NB];
#pragma unroll
      for (int b = 0; b < NB; ++b) r0[b] = round0_step(p0, static_cast<uint32_t>(u * (kStride / 4) + b));
      axpy_values<Io, Mode, V>(
          [&](int i, uint4 (&x)[NB]) {
#pragma unroll
            for (int b = 0; b < NB; ++b) x[b] = gens.words(a, i, r0[b]);
          },
          a, inv, f);
      *reinterpret_cast<typename Io::Vec*>(p + u * kStride) = Io::pack(f);
    }
    if (--tiles == 0) return;
    p += kShape.vecs * kStride;
    p0 = round0_step(p0, kShape.vecs * (kStride / 4));
  }
}

// One unit of the calling thread.
template <class Io, class Mode>
__device__ __forceinline__ void axpy_unit(const UnitRef<Io>& r, const AxpyArgs& a) {
  constexpr int NB = kUnit / 4;
  if (r.rem == 0) return;
  const typename Io::Raw raw = Io::load_unit(r.p, r.rem);
  float f[kUnit];
  Io::unpack_unit(raw, f);
  // a unit's two blocks start at an even one, so they share the high word
  const uint32_t j_hi = static_cast<uint32_t>(r.j0 >> 32);
  const AxpyGens<Mode, false> gens(a, j_hi);
  Round0 r0[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) r0[b] = philox_round0<false>(static_cast<uint32_t>(r.j0 + b));
  axpy_values<Io, Mode, kUnit>(
      [&](int i, uint4 (&x)[NB]) {
#pragma unroll
        for (int b = 0; b < NB; ++b) x[b] = gens.words(a, i, r0[b]);
      },
      a, r.inv, f);
  Io::store_unit(r.p, r.rem, Io::pack_unit(f));
}

// theta[g] <- round(theta[g] + scale * eps_seed[g]) over every segment, or what
// else Mode says. For a scaled storage type (FP8) the noise is added in units of
// the segment's scale: scale * inv_scale[segment].
// A CTA alternates between runs of whole tiles inside one segment (axpy_run)
// and up to a tile's worth of units wherever a segment, the range or a high
// counter word ends (axpy_unit; each thread finds its unit's segment). It waits for
// the kernel before it only when it has read the table.
template <class Io, class Mode>
__device__ __forceinline__ void axpy_pass(const SegDesc* __restrict__ segs, int nseg,
                                          const float* __restrict__ inv_scale, const Split& split,
                                          const AxpyArgs& a) {
  constexpr AxpyShape kShape = axpy_shape<Io, Mode>();
  constexpr uint64_t kTile = axpy_tile_units<Io, Mode>();
  uint64_t q = range_begin(split) * kUnitsPerGranule;
  const uint64_t end = range_end(split) * kUnitsPerGranule;
  int seg = search_segment(segs, 0, nseg, q / kUnitsPerGranule);
  while (q < end) {
    if (q / kUnitsPerGranule >= segs[seg + 1].granule_begin)
      seg = search_segment(segs, seg + 1, nseg, q / kUnitsPerGranule);
    const SegDesc d = segs[seg];
    const uint64_t begin = d.granule_begin * kUnitsPerGranule;
    // where the segment's whole units end
    uint64_t whole = begin + d.numel / kUnit;
    if (whole > end) whole = end;
    if (q + kTile <= whole && blockDim.x == kShape.threads) {
      const uint64_t e = (q - begin) * kUnit, g = d.index_base + e;
      // tiles before the high counter word changes (g passes a multiple of 2^34)
      const uint64_t same_hi = ((((g >> 34) + 1) << 34) - g) / kUnit;
      uint64_t tiles = (whole - q < same_hi ? whole - q : same_hi) / kTile;
      if (tiles > 0) {
        if (tiles > 0x7FFFFFFFu) tiles = 0x7FFFFFFFu;
        const uint64_t mine = threadIdx.x * static_cast<uint64_t>(Io::kVec);
        wait_for_previous();
        axpy_run<Io, Mode>(static_cast<typename Io::Scalar*>(d.data) + e + mine, (g + mine) >> 2,
                            static_cast<uint32_t>(tiles), a, Io::kScaled ? inv_scale[seg] : 1.0f);
        q += tiles * kTile;
        continue;
      }
    }
    const uint64_t stop = q + kTile < end ? q + kTile : end;
    const int last = search_segment(segs, seg, nseg, (stop - 1) / kUnitsPerGranule);
    wait_for_previous();
    // Units of one segment take its entry from registers, which saves a launch
    // 0.2-0.5 us (2^22 bf16 parameters 5.9 -> 5.5 us). Not in the two-step pass and
    // the sums of the 8-element types, bf16 and FP8, where the second loop costs the
    // run above: bf16 2 %; FP8 over 792,680,960 parameters two steps 1118 -> 1126 us,
    // 4 seeds 2116 -> 2126, while launches over 2^18 to 2^22 parameters would gain
    // 0.1-0.4 us with 1 or 2 seeds and lose 0.1-0.2 with 4 or more
    constexpr bool kKeep = Io::kVec != 8 || (!Mode::sum && Mode::seeds == 1);
    bool done = false;
    if constexpr (kKeep) {
      if (seg == last) {
        const float inv = Io::kScaled ? inv_scale[seg] : 1.0f;
#pragma unroll 1
        for (uint64_t u = q + threadIdx.x; u < stop; u += blockDim.x)
          axpy_unit<Io, Mode>(unit_ref<Io>(d, inv, u), a);
        done = true;
      }
    }
    if (!done) {
#pragma unroll 1
      for (uint64_t u = q + threadIdx.x; u < stop; u += blockDim.x) {
        const int s = segment_between(segs, seg, last, u / kUnitsPerGranule);
        axpy_unit<Io, Mode>(unit_ref<Io>(segs[s], Io::kScaled ? inv_scale[s] : 1.0f, u), a);
      }
    }
    __syncwarp();
    q = stop;
    seg = last;
  }
  let_next_start();
}

template <class Io, class Mode>
__global__ void __launch_bounds__(axpy_shape<Io, Mode>().threads, 1)
axpy_noise_kernel(const SegDesc* __restrict__ segs, int nseg, const float* __restrict__ inv_scale,
                  const Split split, const __grid_constant__ AxpyArgs a) {
  axpy_pass<Io, Mode>(segs, nseg, inv_scale, split, a);
}

// The same where every CTA's range is one row at most, one unit per thread: a thread
// has its unit's place before it waits, so that theta's load is all that follows the
// wait. Lane l of a warp loads where segment lo + l begins (a row's 32 units touch at
// most 17 segments) and the threads bisect that by shuffles, which leaves two or three
// dependent loads of the table. axpy_pass looks a row of several segments up behind the
// wait, so a graph of passes over 2 to 4 small tensors ran slower there than through a
// walk along the table, though passes in a stream did not.
// Bound by the latency of one pass. In a graph, us (a walk along the table; axpy_pass ->
// this): 2 fp32 tensors of 300,000 at most, two steps 1.98; 2.39 -> 1.49, perturb 2.06;
// 2.06 -> 1.36; 2 bf16 ones 2.14; 2.43 -> 1.69 and 2.02; 2.14 -> 1.45; 900 bf16 ones of
// 6,000 at most, two steps 3.25 -> 2.27.
// One segment has no lookup to move: up to kRowGranules, where a CTA has 4 warps at
// most, this is the faster one (65,536 fp32 parameters, two steps 2.02 -> 1.36, perturb
// 1.73 -> 1.16); above, a CTA of the next pass that starts early beside one of this pass
// loads some SMs twice, and it is between 20 % faster and 16 % slower (200,000 fp32
// parameters, perturb 1.49 -> 1.73), so one larger segment stays with axpy_pass.
constexpr uint64_t kRowGranules = 8192;
template <class Io, class Mode>
__global__ void __launch_bounds__(axpy_shape<Io, Mode>().threads)
axpy_row_kernel(const SegDesc* __restrict__ segs, int nseg, const float* __restrict__ inv_scale,
                const Split split, const __grid_constant__ AxpyArgs a) {
  const int lane = static_cast<int>(threadIdx.x & 31u);
  const uint64_t last = range_end(split) - 1;
  const uint64_t unit = range_begin(split) * kUnitsPerGranule + threadIdx.x;
  const uint64_t granule = unit / kUnitsPerGranule;
  const uint64_t mine = granule < last ? granule : last;
  int s = 0;
  if (nseg > 1) {
    const uint64_t warp_first = __shfl_sync(0xFFFFFFFFu, mine, 0);
    const int lo = nseg > 32 ? search_segment(segs, 0, nseg, warp_first) : 0;
    const uint64_t begin = lo + lane < nseg ? segs[lo + lane].granule_begin : UINT64_MAX;
#pragma unroll
    for (int step = 16; step > 0; step >>= 1)
      if (__shfl_sync(0xFFFFFFFFu, begin, s + step) <= mine) s += step;
    s += lo;
  }
  UnitRef<Io> r = unit_ref<Io>(segs[s], Io::kScaled ? inv_scale[s] : 1.0f, unit);
  if (granule > last) r.rem = 0;
  wait_for_previous();
  axpy_unit<Io, Mode>(r, a);
  let_next_start();
}

// The same with the segment table in the launch's parameters, for a caller without a
// plan: no copy goes ahead of the kernel in its stream.
template <class Io, class Mode>
__global__ void __launch_bounds__(axpy_shape<Io, Mode>().threads, 1)
axpy_table_kernel(const __grid_constant__ SegTable table, int nseg, const Split split,
                  const __grid_constant__ AxpyArgs a) {
  axpy_pass<Io, Mode>(table.entry, nseg, nullptr, split, a);
}

// Seeds of an update launch are staged in shared memory kSchedRows at a time,
// one row of kRowVecs 16-byte words per seed, filled by the CTA for the
// high counter word j_hi of the units at hand:
//   row[0] = (k0, k1, round 1's k0, tile constant x2)
//   row[1] = (tile constant lo2, coefficient bits, round 1's k1, 0)
//   row[2 .. 5] = round keys of rounds 2..9
// so a seed costs its thread six shared-memory loads instead of deriving its
// key schedule and tile constants. Row kSchedRows is the trailing perturb's.
constexpr int kSchedRows = 128;
constexpr int kRowVecs = 6;
using SchedRow = uint4[kRowVecs];

__device__ __forceinline__ void fill_row(SchedRow& row, uint32_t k0, uint32_t k1, float coeff,
                                         uint32_t j_hi) {
  const PhiloxSched s = philox_sched(static_cast<uint64_t>(k1) << 32 | k0);
  const TileConst t = tile_const(j_hi, s.rk[0], s.rk[3]);
  row[0] = make_uint4(s.rk[0], s.rk[1], s.rk[2], t.x2);
  row[1] = make_uint4(t.lo2, __float_as_uint(coeff), s.rk[3], 0u);
#pragma unroll
  for (int k = 0; k < 4; ++k)
    row[2 + k] = make_uint4(s.rk[4 + 4 * k], s.rk[5 + 4 * k], s.rk[6 + 4 * k], s.rk[7 + 4 * k]);
}

// Round keys of rounds 2..9 held in registers.
struct KeyRegs {
  uint32_t k[16];
  __device__ uint32_t operator[](int i) const { return k[i]; }
};

// Generator of one staged row. kUniformHi: the units at hand share the row's
// high counter word; otherwise the thread's own one is j_hi.
template <bool kUniformHi>
__device__ __forceinline__ SchedGen<KeyRegs> row_gen(const SchedRow& row, uint32_t j_hi) {
  const uint4 r0 = row[0], r1 = row[1];
  KeyRegs kr;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint4 w = row[2 + k];
    kr.k[4 * k] = w.x;
    kr.k[4 * k + 1] = w.y;
    kr.k[4 * k + 2] = w.z;
    kr.k[4 * k + 3] = w.w;
  }
  return {kUniformHi ? TileConst{r0.w, r1.x} : tile_const(j_hi, r0.x, r1.z), r0.y, r0.z, kr};
}

__device__ __forceinline__ float row_coeff(const SchedRow& row) { return __uint_as_float(row[1].y); }

// Which seeds the CTA's rows hold, and for which j_hi.
struct RowState {
  int first;
  uint32_t j_hi;
};

// Makes the rows hold seeds [c0, c0 + kSchedRows) (and the perturb row) for
// j_hi. Called by every thread of the CTA with the same arguments.
template <bool kPerturb>
__device__ __forceinline__ void ensure_rows(SchedRow* s_rows, RowState& rs, const UpdateArgs& args,
                                            int c0, uint32_t j_hi) {
  if (rs.first == c0 && rs.j_hi == j_hi) return;
  __syncthreads();  // every thread is done with the rows held so far
  const int m = args.n - c0 < kSchedRows ? args.n - c0 : kSchedRows;
  for (int k = threadIdx.x; k < m; k += blockDim.x)
    fill_row(s_rows[k], args.key[c0 + k][0], args.key[c0 + k][1], args.coeff[c0 + k], j_hi);
  if (kPerturb && threadIdx.x == blockDim.x - 1)
    fill_row(s_rows[kSchedRows], args.pkey[0], args.pkey[1], args.pscale, j_hi);
  __syncthreads();
  rs.first = c0;
  rs.j_hi = j_hi;
}

// raw <- round(raw + acc) in storage form; acc <- 0.
template <class Io>
__device__ __forceinline__ void apply_acc(typename Io::Raw& raw, float (&acc)[kUnit], float inv) {
  float f[kUnit];
  Io::unpack_unit(raw, f);
#pragma unroll
  for (int k = 0; k < kUnit; ++k) {
    f[k] = add_acc<Io>(f[k], acc[k], inv);
    acc[k] = 0.0f;
  }
  raw = Io::pack_unit(f);
}

// A thread's unit in a fused update launch. Theta stays in registers in
// storage form; generation g adds acc_g = sum_{i in g} c_i eps_i (fp32,
// ascending i) and rounds once, exactly as a separate launch per generation
// would store it (kSingle: one generation, and with kPerturb the next
// generation's first perturb follows, rounded again).
// The loop over the seeds is software-pipelined: seed i + 1's Philox words are
// computed in the same basic block as seed i's transform, so the integer
// multiplies of one seed overlap the MUFU and FP32 work of the other, on
// alternating word buffers (no copies).
template <class Io, bool kUniformHi, bool kSingle, bool kPerturb>
__device__ __forceinline__ void update_unit(typename Io::Scalar* p, int rem, float inv,
                                            uint32_t my_hi, const Round0 (&p0)[kUnit / 4],
                                            uint32_t j_hi, const UpdateArgs& args,
                                            SchedRow* s_rows, RowState& rs) {
  constexpr int NB = kUnit / 4;
  const int n = args.n;
  typename Io::Raw raw = Io::zero_unit();
  if (rem > 0) raw = Io::load_unit(p, rem);
  float acc[kUnit];
#pragma unroll
  for (int k = 0; k < kUnit; ++k) acc[k] = 0.0f;
  auto words = [&](const SchedRow& row, uint4 (&w)[NB]) {
    const auto gen = row_gen<kUniformHi>(row, my_hi);
#pragma unroll
    for (int b = 0; b < NB; ++b) w[b] = gen.block_r0(p0[b]);
  };
  int g = 0;
  int gen_end = kSingle ? n : args.gen_end[0];
#pragma unroll 1
  for (int c0 = 0; c0 < n; c0 += kSchedRows) {
    ensure_rows<kPerturb>(s_rows, rs, args, c0, j_hi);
    const int count = n - c0 < kSchedRows ? n - c0 : kSchedRows;
    if (rem <= 0) continue;
    // seed i of the chunk; at a generation's last seed theta takes the sum
    auto transform = [&](const uint4 (&w)[NB], int i) {
      add_scaled_noise<kUnit>(w, row_coeff(s_rows[i]), acc);
      if constexpr (!kSingle) {
        if (c0 + i + 1 == gen_end) {
          apply_acc<Io>(raw, acc, inv);
          if (++g < args.n_gen) gen_end = args.gen_end[g];
        }
      }
    };
    uint4 x[NB], y[NB];
    words(s_rows[0], x);
    int i = 0;
#pragma unroll 1
    for (; i + 2 < count; i += 2) {
      words(s_rows[i + 1], y);
      transform(x, i);
      words(s_rows[i + 2], x);
      transform(y, i + 1);
    }
    if (i + 1 < count) {
      words(s_rows[i + 1], y);
      transform(x, i);
      transform(y, i + 1);
    } else {
      transform(x, i);
    }
  }
  if (rem <= 0) return;
  if constexpr (kSingle) apply_acc<Io>(raw, acc, inv);
  if constexpr (kPerturb) {
    float f[kUnit];
    Io::unpack_unit(raw, f);
    uint4 x[NB];
    words(s_rows[kSchedRows], x);
    add_scaled_noise<kUnit>(x, row_coeff(s_rows[kSchedRows]) * inv, f);
    raw = Io::pack_unit(f);
  }
  Io::store_unit(p, rem, raw);
}

// Fused update launch (es_update, es_replay, es_update_perturb): for each
// generation g, theta[g] <- round(theta[g] + sum_{i in g} c_i eps_{s_i}[g]),
// then with kPerturb theta <- round(theta + pscale * eps_pseed).
// kSingle: one generation; otherwise args.n_gen generations, never empty.
// A CTA walks its range a row at a time, one unit per thread (8 elements, two
// independent Philox chains, in every storage type): runs of whole rows inside
// one segment from a pointer and a counter that are stepped, and
// single rows, each thread finding its own segment, where a segment, the range
// or a high counter word ends.
// What comes here: one generation of more than 8 seeds, and the passes that several
// generations of a replay share (es_replay), both where update_split_kernel does not
// take them.
// Bound by the generator like the passes above. Measured (3 CTAs of 256 threads on
// grid-stride tiles -> one CTA of 640), ms over 792,680,960 parameters: 16 seeds bf16
// 8.99 -> 8.59 (1.48e12 Gaussians/s), fp32 10.24 -> 8.55 and FP8 9.61 -> 8.59 (their
// seed loops were not pipelined: they took 8 elements in another form), 128 seeds bf16
// 69.0 -> 67.1, 16 seeds + perturb bf16 9.77 -> 9.16. Several generations take 768
// threads, us over 2^24 parameters for 8 generations of 2 seeds (as before; 640 -> 768):
// bf16 228; 205.7 -> 201.8, FP8 236; 206.6 -> 207.0, but fp32 243; 200.4 -> 203.8.
template <bool kSingle>
__host__ __device__ constexpr int update_threads() {
  return kSingle ? 640 : 768;
}

template <class Io, bool kSingle, bool kPerturb>
__global__ void __launch_bounds__(update_threads<kSingle>(), 1)
update_kernel(const SegDesc* __restrict__ segs, int nseg, const float* __restrict__ inv_scale,
              const Split split, const __grid_constant__ UpdateArgs args) {
  constexpr int NB = kUnit / 4;
  __shared__ SchedRow s_rows[kSchedRows + 1];
  RowState rs{-1, 0u};
  const uint32_t row = blockDim.x;
  uint64_t q = range_begin(split) * kUnitsPerGranule;
  const uint64_t end = range_end(split) * kUnitsPerGranule;
  int seg = search_segment(segs, 0, nseg, q / kUnitsPerGranule);
#pragma unroll 1
  while (q < end) {
    if (q / kUnitsPerGranule >= segs[seg + 1].granule_begin)
      seg = search_segment(segs, seg + 1, nseg, q / kUnitsPerGranule);
    const SegDesc d = segs[seg];
    const uint64_t begin = d.granule_begin * kUnitsPerGranule;
    uint64_t whole = begin + d.numel / kUnit;  // where the segment's whole units end
    if (whole > end) whole = end;
    const uint64_t e = (q - begin) * kUnit, index = d.index_base + e;
    const uint32_t j_hi = static_cast<uint32_t>(index >> 34);
    if (q + row <= whole) {
      // rows before the high counter word changes (index passes a multiple of 2^34)
      const uint64_t same_hi = ((((index >> 34) + 1) << 34) - index) / kUnit;
      uint64_t rows = (whole - q < same_hi ? whole - q : same_hi) / row;
      if (rows > 0) {
        q += rows * row;
        typename Io::Scalar* p =
            static_cast<typename Io::Scalar*>(d.data) + e + threadIdx.x * kUnit;
        const float inv = Io::kScaled ? inv_scale[seg] : 1.0f;
        const uint32_t j0 = static_cast<uint32_t>(index >> 2) + threadIdx.x * NB;
        Round0 p0[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) p0[b] = philox_round0<false>(j0 + b);
        ensure_rows<kPerturb>(s_rows, rs, args, 0, j_hi);
        wait_for_previous();
#pragma unroll 1
        for (;;) {
          update_unit<Io, true, kSingle, kPerturb>(p, kUnit, inv, j_hi, p0, j_hi, args, s_rows, rs);
          if (--rows == 0) break;
          p += row * kUnit;
#pragma unroll
          for (int b = 0; b < NB; ++b) p0[b] = round0_step(p0[b], row * NB);
        }
        continue;
      }
    }
    const uint64_t stop = q + row < end ? q + row : end;
    const int last = search_segment(segs, seg, nseg, (stop - 1) / kUnitsPerGranule);
    const uint64_t mine = q + threadIdx.x < stop ? q + threadIdx.x : stop - 1;
    const int s = segment_between(segs, seg, last, mine / kUnitsPerGranule);
    const UnitRef<Io> r = unit_ref<Io>(segs[s], Io::kScaled ? inv_scale[s] : 1.0f, mine);
    const int rem = q + threadIdx.x < stop ? r.rem : 0;
    Round0 p0[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) p0[b] = philox_round0<false>(static_cast<uint32_t>(r.j0 + b));
    const uint32_t my_hi = static_cast<uint32_t>(r.j0 >> 32);
    ensure_rows<kPerturb>(s_rows, rs, args, 0, j_hi);
    wait_for_previous();
    // the staged constants are those of the row's first unit
    if (__syncthreads_and(rem == 0 || my_hi == j_hi))
      update_unit<Io, true, kSingle, kPerturb>(r.p, rem, r.inv, my_hi, p0, j_hi, args, s_rows, rs);
    else
      update_unit<Io, false, kSingle, kPerturb>(r.p, rem, r.inv, my_hi, p0, j_hi, args, s_rows, rs);
    q = stop;
    seg = last;
  }
  let_next_start();
}

// The update of a small set, which leaves most of the GPU's threads without an
// element: the seeds are spread over the warps too. A CTA takes 8 granules (32
// Philox blocks, one per lane) and its warps one seed each at a time; the
// polar forms, scaled, go through shared memory to four of the warps, one per
// element of a block, which add them up in ascending seed order with the same
// operations as update_unit, so the values are the same bits. What bounds it is
// latency: n / kWarps rounds of one block's generation instead of n of two blocks'.
// fp32, us in a graph (the sums' pass or the seed loop -> this): 1,024 parameters 1 seed
// 1.36 -> 1.12, 32 seeds 6.6 -> 2.4, 128 seeds 22.5 -> 8.6; 65,536 parameters 1.53 ->
// 1.57, 7.0 -> 6.0, 22.4 -> 20.5, and 8 seeds 2.9 -> 2.2. It generates one block per
// thread where the others overlap two, so it loses once the GPU is full, at a size that
// depends on the population: 1 and 2 seeds are even at 65,536 parameters, 8 seeds at
// 98,304 (2.9 -> 2.8), 16 and 32 at 81,920 (7.1 -> 7.2); 128 seeds gain there yet (30.3,
// where the loop's rows just miss its CTAs, -> 25.2) and lose at 98,304 (22.4 -> 29.7).
// kSplitMaxGranules, 69,632 parameters, is one line for all: up to it only 1 seed loses,
// 0.06 us (bf16 0.11), and 32 gain 7.1 -> 6.0, 128 22.3 -> 20.5.
// A launch of more than kSplitSeeds seeds does not come here whatever its size. That
// is what SplitArgs holds and no break-even: 129 seeds take the seed loop 23.3 us over
// 1,000 parameters, where 128 take 8.7, and 22.8 against 20.5 over 65,536.
// A CTA of 32 warps, 32 seeds at a time, is taken for more than 8 while every CTA has
// one of the GPU's 152 SMs to itself (19,456 parameters, 128 seeds 13.1 with 8 warps ->
// 9.1). With two on an SM it still gains from 32 seeds on (32,768 parameters 13.7 ->
// 12.2) and loses with 16 (2.59 -> 2.63); at 65,536 it loses with any (20.5 -> 23.8).
constexpr uint64_t kSplitMaxGranules = 4352;
constexpr uint64_t kSplitWideGranules = 152 * 8;
constexpr int kSplitSeeds = 128;
struct SplitArgs {
  int n, n_gen, perturb;  // as UpdateArgs
  float pscale;
  uint32_t pkey[2];
  uint8_t gen_end[kSplitSeeds];
  uint32_t key[kSplitSeeds][2];
  float coeff[kSplitSeeds];
};
constexpr int kSplitGranules = 32 * 4 / kGranule;
// One warp's scaled polar forms: -(c r) of both pairs, then cos and sin of each.
using SplitForms = float[6][32];

template <class Io, int kWarps>
__global__ void __launch_bounds__(32 * kWarps)
update_split_kernel(const SegDesc* __restrict__ segs, int nseg, const float* __restrict__ inv_scale,
                    uint64_t granules, const __grid_constant__ SplitArgs args) {
  __shared__ SplitForms s_forms[2][kWarps];
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  const uint64_t first = blockIdx.x * static_cast<uint64_t>(kSplitGranules);
  const uint64_t end = first + kSplitGranules < granules ? first + kSplitGranules : granules;
  // the lane's block: 4 elements at e in its segment
  const int seg0 = search_segment(segs, 0, nseg, first);
  const int seg1 = search_segment(segs, seg0, nseg, end - 1);
  const uint64_t mine = first + lane / 4 < end ? first + lane / 4 : end - 1;
  const int seg = segment_between(segs, seg0, seg1, mine);
  const SegDesc d = segs[seg];
  const uint64_t e = (mine - d.granule_begin) * kGranule + lane % 4 * 4;
  const float inv = Io::kScaled ? inv_scale[seg] : 1.0f;
  const uint64_t j = (d.index_base + e) >> 2;
  // warps 0 .. 3 own element `warp` of each block
  const bool owner = warp < 4 && first + lane / 4 < end && e + warp < d.numel;
  typename Io::Scalar* const p = static_cast<typename Io::Scalar*>(d.data) + e + warp;
  float theta = 0.0f, acc = 0.0f;
  int g = 0;
  const int items = args.n + args.perturb;  // the perturb comes last
#pragma unroll 1
  for (int i0 = 0, buf = 0; i0 < items; i0 += kWarps, buf ^= 1) {
    const int i = i0 + warp;
    if (i < items) {
      const bool last = i == args.n;
      const PhiloxKey key = last ? PhiloxKey{args.pkey[0], args.pkey[1]}
                                 : PhiloxKey{args.key[i][0], args.key[i][1]};
      const float scale = last ? args.pscale * inv : args.coeff[i];
      const uint4 x[1] = {philox_block(j, key)};
      Polar2 pp[1];
      polar_from_words<1>(x, pp);
      const float2 sr = __fmul2_rn(make_float2(-scale, -scale), pp[0].r);
      SplitForms& f = s_forms[buf][warp];
      f[0][lane] = sr.x;
      f[1][lane] = sr.y;
      f[2][lane] = pp[0].c.x;
      f[3][lane] = pp[0].s.x;
      f[4][lane] = pp[0].c.y;
      f[5][lane] = pp[0].s.y;
    }
    if (i0 == 0) {
      wait_for_previous();
      if (owner) theta = Io::value(*p);
    }
    __syncthreads();
    if (warp >= 4) continue;
    const int m = items - i0 < kWarps ? items - i0 : kWarps;
#pragma unroll 8
    for (int k = 0; k < kWarps; ++k) {
      if (k >= m) break;
      const SplitForms& f = s_forms[buf][k];
      const float sr = f[warp / 2][lane], t = f[2 + warp][lane];
      if (i0 + k == args.n) {
        theta = Io::value(Io::store(fmaf(sr, t, theta)));
      } else {
        acc = fmaf(sr, t, acc);
        if (i0 + k + 1 == args.gen_end[g]) {
          theta = Io::value(Io::store(add_acc<Io>(theta, acc, inv)));
          acc = 0.0f;
          if (g + 1 < args.n_gen) ++g;
        }
      }
    }
  }
  if (owner) *p = Io::store(theta);
  let_next_start();
}

// es_noise_fill. `out` is cut into aligned 16-byte groups of 4 floats, and group
// m lies `lead` floats before out[4m]; its values come from one Philox block
// (kShift 0) or from the last 4 - kShift values of one block and the first
// kShift of the next, depending on how index_base and out's alignment meet. A
// warp takes a contiguous run of rows of 32 groups; each lane generates one
// block per row and gets the values of the block before from the lane below
// (lane 0: from lane 31's block of the row before), so every block is generated
// once and every store is a coalesced 16 bytes. Only the first and the last
// group, which may reach beyond [0, n), store element by element.
// Bound by the generator, and by the stores' bandwidth not far behind (500,000,000
// aligned floats run at 5.76 TB/s). 50,000,003 floats from an unaligned index 58.4 us
// (4-byte stores, every block through the general rounds) -> 40.3; 50,000,000
// aligned 44.3 (256-thread CTAs, one block at a time) -> 36.8, 500,000,000 418 -> 347.
// 512 to 768 threads and 2 pairs of rows per loop are within 2 %; 1024 threads lose 8 %.
struct FillArgs {
  PhiloxSched sched;
  uint64_t j_first;   // block of group 0 (kShift > 0: the block it ends in)
  uint64_t groups;
  uint64_t per_warp;  // groups of one warp: a row, or a multiple of 64
  uint64_t n;
  int lead;
};
constexpr int kFillThreads = 768;
// Groups of a row on its own (noise_row_kernel).
__host__ __device__ constexpr uint64_t fill_row_groups(int shift) { return shift != 0 ? 31 : 32; }

__device__ __forceinline__ float4 polar_values(const Polar2& p) {
  const float2 lo = __fmul2_rn(make_float2(-p.r.x, -p.r.x), make_float2(p.c.x, p.s.x));
  const float2 hi = __fmul2_rn(make_float2(-p.r.y, -p.r.y), make_float2(p.c.y, p.s.y));
  return make_float4(lo.x, lo.y, hi.x, hi.y);
}

// The group that ends in the calling lane's block `cur`: before is the lane's
// block of the row before (only lane 31's is used).
template <int kShift>
__device__ __forceinline__ float4 fill_group(const float4& cur, const float4& before, uint32_t lane) {
  if constexpr (kShift == 0) {
    return cur;
  } else {
    const bool top = lane == 31;
    const uint32_t from = (lane + 31) & 31;
    const float w = __shfl_sync(0xFFFFFFFFu, top ? before.w : cur.w, from);
    if constexpr (kShift == 3) return make_float4(w, cur.x, cur.y, cur.z);
    const float z = __shfl_sync(0xFFFFFFFFu, top ? before.z : cur.z, from);
    if constexpr (kShift == 2) return make_float4(z, w, cur.x, cur.y);
    const float y = __shfl_sync(0xFFFFFFFFu, top ? before.y : cur.y, from);
    return make_float4(y, z, w, cur.x);
  }
}

// Values of NB blocks from round 0's products.
template <int NB, class Gen>
__device__ __forceinline__ void fill_values(const Gen& gen, const Round0 (&p0)[NB],
                                            float4 (&v)[NB]) {
  uint4 x[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) x[b] = gen.block_r0(p0[b]);
  Polar2 p[NB];
  polar_from_words<NB>(x, p);
#pragma unroll
  for (int b = 0; b < NB; ++b) v[b] = polar_values(p[b]);
}

template <int kShift>
__global__ void __launch_bounds__(kFillThreads, 1)
noise_fill_kernel(const __grid_constant__ FillArgs a, float* __restrict__ out) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t warp =
      blockIdx.x * static_cast<uint64_t>(blockDim.x / 32) + threadIdx.x / 32;
  uint64_t m = warp * a.per_warp;
  const uint64_t end = m + a.per_warp < a.groups ? m + a.per_warp : a.groups;
  // where the warp's groups that lie inside [0, n) end
  const uint64_t inside = (a.n + a.lead) / 4 < end ? (a.n + a.lead) / 4 : end;
#pragma unroll 1
  while (m < end) {
    const uint64_t j = a.j_first + m;
    const uint32_t j_hi = static_cast<uint32_t>(j >> 32);
    // Pairs of rows with whole groups (not group 0 where it is cut off) and one
    // high counter word
    const uint64_t same_hi = ((static_cast<uint64_t>(j_hi) + 1) << 32) - j;
    const uint64_t limit = m >= inside || (m == 0 && a.lead != 0) ? 0 : inside - m;
    const uint64_t pairs = (limit < same_hi ? limit : same_hi) / 64;
    if (pairs > 0) {
      float4 before = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if constexpr (kShift != 0) {
        const auto gen = sched_gen<false>(a.sched, static_cast<uint32_t>((j - 1) >> 32));
        const Round0 p0[1] = {philox_round0<false>(static_cast<uint32_t>(j - 1))};
        float4 v[1];
        fill_values<1>(gen, p0, v);
        before = v[0];
      }
      const auto gen = sched_gen<true>(a.sched, j_hi);
      Round0 p0 = philox_round0<true>(static_cast<uint32_t>(j) + lane);
      float4* o = reinterpret_cast<float4*>(out + 4 * m - a.lead) + lane;
      wait_for_previous();
#pragma unroll 2
      for (uint32_t i = static_cast<uint32_t>(pairs); i > 0; --i) {
        const Round0 rows[2] = {p0, round0_step(p0, 32u)};
        float4 v[2];
        fill_values<2>(gen, rows, v);
        __stcs(o, fill_group<kShift>(v[0], before, lane));
        __stcs(o + 32, fill_group<kShift>(v[1], v[0], lane));
        if constexpr (kShift != 0) before = v[1];
        o += 64;
        p0 = round0_step(p0, 64u);
      }
      m += 64 * pairs;
      continue;
    }
    // one row: each lane its own high word and bounds, and the block before it
    constexpr int NB = kShift != 0 ? 2 : 1;
    float4 v[2];
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const uint64_t mine = b == 0 ? j + lane : j - 1;
      const auto gen = sched_gen<false>(a.sched, static_cast<uint32_t>(mine >> 32));
      const Round0 p0[1] = {philox_round0<false>(static_cast<uint32_t>(mine))};
      float4 w[1];
      fill_values<1>(gen, p0, w);
      v[b] = w[0];
    }
    const float4 q = fill_group<kShift>(v[0], v[NB - 1], lane);
    const uint64_t k = 4 * (m + lane) - a.lead;  // wraps below zero only in group 0
    wait_for_previous();
    const float f[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (m + lane < end && k + i < a.n) out[k + i] = f[i];
    m += 32;
  }
  let_next_start();
}

// The same where one row per warp is enough for `out` (2 CTAs per SM: 933,888 aligned
// floats), each lane with its own high word and bounds. With a shift lane 0 generates
// the block before the row's first, for lane 1, and has no group of its own;
// noise_fill_kernel has every lane generate that block, which cost unaligned fills of
// this size more than one thread per block had. Bound by one block's latency and the
// launch. In a graph, us (one thread per block; noise_fill_kernel -> this): unaligned
// 1 float 0.87; 1.24 -> 0.83, 450,000 1.65; 2.10 -> 1.36, 800,000 2.22; 2.38 -> 1.85;
// aligned 450,000 1.90; 1.61 -> 1.24.
template <int kShift>
__global__ void __launch_bounds__(kFillThreads)
noise_row_kernel(const __grid_constant__ FillArgs a, float* __restrict__ out) {
  constexpr uint32_t kBefore = kShift != 0 ? 1 : 0;
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t warp =
      blockIdx.x * static_cast<uint64_t>(blockDim.x / 32) + threadIdx.x / 32;
  const uint64_t m = warp * fill_row_groups(kShift);
  if (m < a.groups) {
    const uint64_t group = m + lane - kBefore, j = a.j_first + group;
    const auto gen = sched_gen<false>(a.sched, static_cast<uint32_t>(j >> 32));
    const Round0 p0[1] = {philox_round0<false>(static_cast<uint32_t>(j))};
    float4 v[1];
    fill_values<1>(gen, p0, v);
    const float4 q = fill_group<kShift>(v[0], v[0], lane);
    const uint64_t k = 4 * group - a.lead;  // wraps below zero only in group 0
    wait_for_previous();
    const float f[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if ((kShift == 0 || lane > 0) && group < a.groups && k + i < a.n) out[k + i] = f[i];
  }
  let_next_start();
}

// out[4t .. 4t+3] = Philox words of block block_base + t. Block j goes
// through one of the four implementations of the rounds by j mod 4: the
// general one (philox_block), the one with per-tile constants (philox_tile),
// and the scheduled-key one the streaming kernels use, with high/low product
// pairs in the first two rounds (philox_block_rk), or with 64-bit-result
// products throughout and round 0's product stepped from that of a lower
// counter word by 64-bit additions (round0_step, philox_block_r0). They give
// identical words, and this lets a bit-exact check of this output cover all
// four.
__global__ void __launch_bounds__(kBlockThreads)
noise_bits_kernel(uint64_t block_base, uint64_t nblocks, const __grid_constant__ PhiloxSched sched,
                  uint4* __restrict__ out) {
  const PhiloxKey key{sched.rk[0], sched.rk[1]};
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
  for (uint64_t t = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; t < nblocks;
       t += stride) {
    const uint64_t j = block_base + t;
    const uint32_t j_lo = static_cast<uint32_t>(j), j_hi = static_cast<uint32_t>(j >> 32);
    const TileConst tc = tile_const(j_hi, sched.rk[0], sched.rk[3]);
    switch (j & 3) {
      case 0: out[t] = philox_block(j, key); break;
      case 1: out[t] = philox_block_tile(j_lo, philox_tile(j_hi, key)); break;
      case 2: out[t] = philox_block_rk<false>(j_lo, tc, sched.rk[1], sched.rk[2], sched.rk + 4); break;
      default: {
        // from j_lo rounded down to a multiple of 2^11, d = j_lo mod 2^11 (no wrap)
        const Round0 p0 = round0_step(philox_round0<true>(j_lo & ~0x7FFu), j_lo & 0x7FFu);
        out[t] = philox_block_r0<true>(p0, tc, sched.rk[1], sched.rk[2], sched.rk + 4);
      }
    }
  }
}

// out[2k], out[2k+1] = Box-Muller pair of words[2k], words[2k+1].
__global__ void __launch_bounds__(kBlockThreads)
box_muller_kernel(const uint2* __restrict__ words, uint64_t npairs, float2* __restrict__ out) {
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
  for (uint64_t k = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; k < npairs;
       k += stride) {
    const uint2 w = words[k];
    out[k] = box_muller(w.x, w.y);
  }
}

// Resident CTAs of one kernel on one device (SMs x CTAs per SM), looked up
// with the occupancy calculator on the kernel's first launch on that device
// and kept, so later launches make no query beyond cudaGetDevice.
struct GridEntry {
  const void* kernel;
  int device;
  int ctas;
};
constexpr int kGridCacheSize = 512;
std::mutex g_grid_mutex;
GridEntry g_grid_cache[kGridCacheSize];
int g_grid_used = 0;

int resident_ctas(const void* kernel, int threads, int dev) {
  {
    std::lock_guard<std::mutex> lock(g_grid_mutex);
    for (int k = 0; k < g_grid_used; ++k)
      if (g_grid_cache[k].kernel == kernel && g_grid_cache[k].device == dev)
        return g_grid_cache[k].ctas;
  }
  int sms = 0, per_sm = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0);
  if (sms < 1) sms = 1;
  if (per_sm < 1) per_sm = 1;
  const int ctas = sms * per_sm;
  std::lock_guard<std::mutex> lock(g_grid_mutex);
  if (g_grid_used < kGridCacheSize) g_grid_cache[g_grid_used++] = GridEntry{kernel, dev, ctas};
  return ctas;
}

// Persistent grid: every SM filled to the kernel's occupancy, never more
// CTAs than tiles.
template <class K>
int persistent_grid(K kernel, uint64_t work_items) {
  int dev = 0;
  cudaGetDevice(&dev);
  uint64_t grid = static_cast<uint64_t>(resident_ctas(reinterpret_cast<const void*>(kernel), kBlockThreads, dev));
  if (work_items < grid) grid = work_items;
  return grid < 1 ? 1 : static_cast<int>(grid);
}

// A streaming launch: its division, grid and block size.
struct Launch {
  Split split;
  int grid, block;
};

// One range per resident CTA and no less than a warp's units; long ranges in
// whole 8-granule pieces (256 bytes of bf16), so that they meet at cache-line
// boundaries.
// Where the ranges are shorter than `whole_block` units the block shrinks to
// what they need, in rows of equal length (a multiple of 128 threads above
// 128: each SM sub-partition then holds as many warps as the others; 448 and
// 576 threads measured 10 % slower than 384 and 512).
Launch make_launch(const void* kernel, int threads, uint64_t whole_block, uint64_t granules) {
  int dev = 0;
  cudaGetDevice(&dev);
  const uint64_t ctas = static_cast<uint64_t>(resident_ctas(kernel, threads, dev));
  uint64_t per = (granules + ctas - 1) / ctas;
  if (per >= 512) per = (per + 7) / 8 * 8;
  if (per < 32 / kUnitsPerGranule) per = 32 / kUnitsPerGranule;
  Launch l;
  l.split = Split{granules, per};
  l.grid = static_cast<int>((granules + per - 1) / per);
  l.block = threads;
  const uint64_t units = per * kUnitsPerGranule;
  if (units < whole_block) {
    const uint64_t rows = (units + threads - 1) / threads;
    const uint64_t want = (units + rows - 1) / rows;
    const uint64_t step = want > 128 ? 128 : 32;
    const uint64_t block = (want + step - 1) / step * step;
    l.block = static_cast<int>(block < static_cast<uint64_t>(threads) ? block : threads);
  }
  return l;
}

// Launches a kernel that calls let_next_start and wait_for_previous; `early`
// allows it to start before the kernel before it in the stream has ended.
template <class... P, class... A>
cudaError_t launch_early(void (*kernel)(P...), int grid, int block, bool early, cudaStream_t stream,
                         const A&... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = early ? 1 : 0;
  cudaLaunchConfig_t config{};
  config.gridDim = dim3(static_cast<unsigned>(grid));
  config.blockDim = dim3(static_cast<unsigned>(block));
  config.stream = stream;
  config.attrs = &attr;
  config.numAttrs = 1;
  const cudaError_t err = cudaLaunchKernelEx(&config, kernel, P(args)...);
  const cudaError_t last = cudaGetLastError();
  return err != cudaSuccess ? err : last;
}

template <class Io, class Mode>
cudaError_t launch_axpy_io(const PlanView& plan, const AxpyArgs& a, cudaStream_t stream) {
  auto k = axpy_noise_kernel<Io, Mode>;
  const Launch l = make_launch(reinterpret_cast<const void*>(k), axpy_shape<Io, Mode>().threads,
                               axpy_tile_units<Io, Mode>(), plan.granules);
  if constexpr (!Mode::sum)
    if (l.split.per_cta * kUnitsPerGranule <= static_cast<uint64_t>(l.block) &&
        (plan.nseg > 1 || plan.granules <= kRowGranules))
      return launch_early(axpy_row_kernel<Io, Mode>, l.grid, l.block, plan.early, stream, plan.segs,
                          plan.nseg, plan.inv_scale, l.split, a);
  return launch_early(k, l.grid, l.block, plan.early, stream, plan.segs, plan.nseg, plan.inv_scale,
                      l.split, a);
}

template <class Mode>
cudaError_t launch_axpy(const PlanView& plan, const AxpyArgs& a, cudaStream_t stream) {
  if (plan.dtype == ES_BF16) return launch_axpy_io<Bf16Io, Mode>(plan, a, stream);
  if (plan.dtype == ES_FP8_E4M3) return launch_axpy_io<Fp8Io, Mode>(plan, a, stream);
  return launch_axpy_io<F32Io, Mode>(plan, a, stream);
}

}  // namespace

cudaError_t launch_axpy_noise(const PlanView& plan, uint64_t seed, float scale,
                              cudaStream_t stream) {
  AxpyArgs a{};
  a.seed[0] = philox_sched(seed);
  a.scale[0] = scale;
  return launch_axpy<AxpyOne>(plan, a, stream);
}

template <class Io>
cudaError_t launch_table_io(const SegTable& table, int nseg, const AxpyArgs& a,
                            cudaStream_t stream) {
  auto k = axpy_table_kernel<Io, AxpyOne>;
  const Launch l = make_launch(reinterpret_cast<const void*>(k), axpy_shape<Io, AxpyOne>().threads,
                               axpy_tile_units<Io, AxpyOne>(), table.entry[nseg].granule_begin);
  return launch_early(k, l.grid, l.block, true, stream, table, nseg, l.split, a);
}

cudaError_t launch_axpy_table(const SegTable& table, int nseg, es_dtype_t dtype, uint64_t seed,
                              float scale, cudaStream_t stream) {
  AxpyArgs a{};
  a.seed[0] = philox_sched(seed);
  a.scale[0] = scale;
  return dtype == ES_BF16 ? launch_table_io<Bf16Io>(table, nseg, a, stream)
                          : launch_table_io<F32Io>(table, nseg, a, stream);
}

cudaError_t launch_axpy_noise2(const PlanView& plan, uint64_t seed, float scale, uint64_t seed2,
                               float scale2, cudaStream_t stream) {
  AxpyArgs a{};
  a.seed[0] = philox_sched(seed);
  a.seed[1] = philox_sched(seed2);
  a.scale[0] = scale;
  a.scale[1] = scale2;
  return seed == seed2 ? launch_axpy<AxpyFlip>(plan, a, stream)
                       : launch_axpy<AxpyTwo>(plan, a, stream);
}

template <class Io, bool kSingle, bool kPerturb>
cudaError_t launch_update_io(const PlanView& plan, const UpdateArgs& args, cudaStream_t stream) {
  auto k = update_kernel<Io, kSingle, kPerturb>;
  constexpr int kThreads = update_threads<kSingle>();
  const Launch l = make_launch(reinterpret_cast<const void*>(k), kThreads, 4 * kThreads, plan.granules);
  return launch_early(k, l.grid, l.block, plan.early, stream, plan.segs, plan.nseg, plan.inv_scale,
                      l.split, args);
}

template <class Io>
cudaError_t launch_update_dtype(const PlanView& plan, const UpdateArgs& args, cudaStream_t stream) {
  if (args.n_gen > 1) return launch_update_io<Io, false, false>(plan, args, stream);
  return args.perturb ? launch_update_io<Io, true, true>(plan, args, stream)
                      : launch_update_io<Io, true, false>(plan, args, stream);
}

template <class Io, int kWarps>
cudaError_t launch_split_warps(const PlanView& plan, const SplitArgs& args, cudaStream_t stream) {
  return launch_early(update_split_kernel<Io, kWarps>,
                      static_cast<int>((plan.granules + kSplitGranules - 1) / kSplitGranules),
                      32 * kWarps, plan.early, stream, plan.segs, plan.nseg, plan.inv_scale,
                      plan.granules, args);
}

template <class Io>
cudaError_t launch_split_io(const PlanView& plan, const SplitArgs& args, cudaStream_t stream) {
  if (args.n + args.perturb > 8 && plan.granules <= kSplitWideGranules)
    return launch_split_warps<Io, 32>(plan, args, stream);
  return launch_split_warps<Io, 8>(plan, args, stream);
}

cudaError_t launch_update_split(const PlanView& plan, const UpdateArgs& args, cudaStream_t stream) {
  SplitArgs a;
  a.n = args.n;
  a.n_gen = args.n_gen;
  a.perturb = args.perturb;
  a.pscale = args.pscale;
  a.pkey[0] = args.pkey[0];
  a.pkey[1] = args.pkey[1];
  for (int g = 0; g < args.n_gen; ++g) a.gen_end[g] = static_cast<uint8_t>(args.gen_end[g]);
  for (int i = 0; i < args.n; ++i) {
    a.key[i][0] = args.key[i][0];
    a.key[i][1] = args.key[i][1];
    a.coeff[i] = args.coeff[i];
  }
  if (plan.dtype == ES_BF16) return launch_split_io<Bf16Io>(plan, a, stream);
  if (plan.dtype == ES_FP8_E4M3) return launch_split_io<Fp8Io>(plan, a, stream);
  return launch_split_io<F32Io>(plan, a, stream);
}

template <int N>
cudaError_t launch_sum_of(const PlanView& plan, const AxpyArgs& a, bool perturb,
                          cudaStream_t stream) {
  return perturb ? launch_axpy<AxpySumPerturb<N>>(plan, a, stream)
                 : launch_axpy<AxpySum<N>>(plan, a, stream);
}

cudaError_t launch_sum(const PlanView& plan, const UpdateArgs& args, cudaStream_t stream) {
  AxpyArgs a{};
  for (int i = 0; i < args.n; ++i) {
    a.seed[i] = philox_sched(static_cast<uint64_t>(args.key[i][1]) << 32 | args.key[i][0]);
    a.scale[i] = args.coeff[i];
  }
  if (args.perturb) {
    a.seed[args.n] = philox_sched(static_cast<uint64_t>(args.pkey[1]) << 32 | args.pkey[0]);
    a.scale[args.n] = args.pscale;
  }
  const bool p = args.perturb != 0;
  switch (args.n) {
    case 1: return launch_sum_of<1>(plan, a, p, stream);
    case 2: return launch_sum_of<2>(plan, a, p, stream);
    case 3: return launch_sum_of<3>(plan, a, p, stream);
    case 4: return launch_sum_of<4>(plan, a, p, stream);
    case 5: return launch_sum_of<5>(plan, a, p, stream);
    case 6: return launch_sum_of<6>(plan, a, p, stream);
    case 7: return launch_sum_of<7>(plan, a, p, stream);
    default: return launch_sum_of<8>(plan, a, p, stream);
  }
}

cudaError_t launch_update(const PlanView& plan, const UpdateArgs& args, cudaStream_t stream) {
  if (args.n <= kSplitSeeds && plan.granules <= kSplitMaxGranules)
    return launch_update_split(plan, args, stream);
  if (args.n_gen == 1 && args.n <= kMaxSum) return launch_sum(plan, args, stream);
  if (plan.dtype == ES_BF16) return launch_update_dtype<Bf16Io>(plan, args, stream);
  if (plan.dtype == ES_FP8_E4M3) return launch_update_dtype<Fp8Io>(plan, args, stream);
  return launch_update_dtype<F32Io>(plan, args, stream);
}

cudaError_t launch_noise_bits(uint64_t seed, uint64_t block_base, uint64_t nblocks,
                              uint32_t* out, cudaStream_t stream) {
  const uint64_t ctas = (nblocks + kBlockThreads - 1) / kBlockThreads;
  const int grid = persistent_grid(noise_bits_kernel, ctas);
  noise_bits_kernel<<<grid, kBlockThreads, 0, stream>>>(block_base, nblocks, philox_sched(seed),
                                                        reinterpret_cast<uint4*>(out));
  return cudaGetLastError();
}

cudaError_t launch_box_muller(const uint32_t* words, uint64_t npairs, float* out,
                              cudaStream_t stream) {
  const uint64_t ctas = (npairs + kBlockThreads - 1) / kBlockThreads;
  const int grid = persistent_grid(box_muller_kernel, ctas);
  box_muller_kernel<<<grid, kBlockThreads, 0, stream>>>(reinterpret_cast<const uint2*>(words),
                                                        npairs, reinterpret_cast<float2*>(out));
  return cudaGetLastError();
}

cudaError_t launch_noise_fill(uint64_t seed, uint64_t index_base, uint64_t n, float* out,
                              cudaStream_t stream) {
  FillArgs a;
  a.sched = philox_sched(seed);
  a.n = n;
  a.lead = static_cast<int>(reinterpret_cast<uintptr_t>(out) / 4 % 4);
  const int shift = static_cast<int>((index_base - a.lead) & 3u);
  // the block of group 0's first element (-1, i.e. 2^64 - 1, if that element
  // comes before index 0: its values are not stored)
  a.j_first = index_base / 4 - (index_base % 4 < static_cast<uint64_t>(a.lead) ? 1u : 0u) +
              (shift != 0 ? 1u : 0u);
  a.groups = n / 4 + (n % 4 + a.lead + 3) / 4;
  using Kernel = void (*)(FillArgs, float*);
  static constexpr Kernel kRow[4] = {noise_row_kernel<0>, noise_row_kernel<1>, noise_row_kernel<2>,
                                     noise_row_kernel<3>};
  static constexpr Kernel kFill[4] = {noise_fill_kernel<0>, noise_fill_kernel<1>,
                                      noise_fill_kernel<2>, noise_fill_kernel<3>};
  int dev = 0;
  cudaGetDevice(&dev);
  auto resident = [&](Kernel k) {
    return static_cast<uint64_t>(
        resident_ctas(reinterpret_cast<const void*>(k), kFillThreads, dev));
  };
  constexpr uint64_t kWarps = kFillThreads / 32;
  Kernel k = kRow[shift];
  uint64_t ctas = resident(k);
  a.per_warp = fill_row_groups(shift);
  if ((a.groups + a.per_warp - 1) / a.per_warp > ctas * kWarps) {
    k = kFill[shift];
    ctas = resident(k);
    const uint64_t rows = ((a.groups + 31) / 32 + ctas * kWarps - 1) / (ctas * kWarps);
    a.per_warp = (rows + 1) / 2 * 64;
  }
  const uint64_t warps = (a.groups + a.per_warp - 1) / a.per_warp;
  // spread over the SMs, whole sets of 4 warps (one per SM sub-partition) above 4
  uint64_t per_cta = (warps + ctas - 1) / ctas;
  if (per_cta > 4) per_cta = (per_cta + 3) / 4 * 4;
  return launch_early(k, static_cast<int>((warps + per_cta - 1) / per_cta),
                      static_cast<int>(32 * per_cta), true, stream, a, out);
}

}  // namespace esopt
