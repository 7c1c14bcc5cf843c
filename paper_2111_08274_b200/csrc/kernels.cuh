// sm_100a kernels of the HADFL round: initial model (K0), batched heterogeneity-aware local
// update (K1; Eq. 3 / Algorithm 1), fused weighted aggregation with write-back (K2; Eq. 5),
// the mix of a received model into the receivers' own (Section "Model aggregation and
// fault-tolerant"), per-replica statistics (K3), and the fused round (K1 + K2 + global
// synchronisation + K3 in one pass over the arena).
//
// All of them stream rows of one [N][stride] arena.  A "column group" is four consecutive
// parameters (one Philox block); a thread holds a "pack" of a row - 16 bytes of w in K2 / K3,
// eight parameters in K1 and the fused round - and walks over the rows, so that
//   - accesses of a warp are contiguous (512 bytes per 128-bit load instruction),
//   - several independent row loads are in flight per thread before the first dependent use
//     (loads fill raw packs; widening bf16 to fp32 happens where the values are used),
//   - every thread does the same amount of arithmetic whatever the per-device step counts are
//     (the kernel-level answer to the straggler problem the paper is about), and
//   - the arithmetic order per element is fixed, hence results are reproducible bit for bit.
// None of this is a dense contraction, so there is no tensor-core path: the bound is HBM
// bandwidth, except for the local update with several steps per device, where instruction issue
// (the integer multiplies of Philox, Box-Muller on the special-function unit) binds.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "debug_check.cuh"
#include "philox.cuh"

namespace hadfl {

constexpr int kMaxDevices = 32;
constexpr int kThreads = 256;

// ------------------------------------------------------------------------------------------
// Storage access by element and by column group (used by the initial-model kernel and by the
// ragged last pack of a row).
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ void st_group(float *row, int64_t g, float4 v) {
  if (!access_ok(row + 4 * g, 16)) return;
  *reinterpret_cast<float4 *>(row + 4 * g) = v;
}
__device__ __forceinline__ void st_group(__nv_bfloat16 *row, int64_t g, float4 v) {
  if (!access_ok(row + 4 * g, 8)) return;
  const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y);
  const __nv_bfloat162 hi = __floats2bfloat162_rn(v.z, v.w);
  uint2 raw;
  raw.x = *reinterpret_cast<const uint32_t *>(&lo);
  raw.y = *reinterpret_cast<const uint32_t *>(&hi);
  *reinterpret_cast<uint2 *>(row + 4 * g) = raw;
}
__device__ __forceinline__ void st_elem(float *row, int64_t p, float v) {
  if (access_ok(row + p, 4)) row[p] = v;
}
__device__ __forceinline__ void st_elem(__nv_bfloat16 *row, int64_t p, float v) {
  if (access_ok(row + p, 2)) row[p] = __float2bfloat16_rn(v);
}

// ------------------------------------------------------------------------------------------
// Packs: E consecutive parameters held by one thread (E = 4 or 8).  fp32: E/4 128-bit accesses;
// bf16: one 64-bit (E = 4) or 128-bit (E = 8) access.  A pack of 8 is two column groups, i.e.
// two Philox blocks.  `live` < E only in the ragged last pack of a row.
// ------------------------------------------------------------------------------------------
template <typename WT>
struct Pack16 {  // the pack that is 16 bytes of storage
  static constexpr int E = sizeof(WT) == 2 ? 8 : 4;
};

template <int E>
__device__ __forceinline__ void st_pack(float *row, int64_t p, const float (&v)[E]) {
  if (!access_ok(row + E * p, 4 * E)) return;
#pragma unroll
  for (int i = 0; i < E / 4; ++i)
    *reinterpret_cast<float4 *>(row + E * p + 4 * i) =
        make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
}
__device__ __forceinline__ void bf16x2_to_floats(uint32_t raw, float &lo, float &hi) {
  lo = __uint_as_float(raw << 16);
  hi = __uint_as_float(raw & 0xFFFF0000u);
}
__device__ __forceinline__ uint32_t floats_to_bf16x2(float lo, float hi) {
  const __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t *>(&t);
}
template <int E>
__device__ __forceinline__ void st_pack(__nv_bfloat16 *row, int64_t p, const float (&v)[E]) {
  if (!access_ok(row + E * p, 2 * E)) return;
  if (E == 8) {
    uint4 raw;
    raw.x = floats_to_bf16x2(v[0], v[1]);
    raw.y = floats_to_bf16x2(v[2], v[3]);
    raw.z = floats_to_bf16x2(v[E - 4], v[E - 3]);
    raw.w = floats_to_bf16x2(v[E - 2], v[E - 1]);
    *reinterpret_cast<uint4 *>(row + 8 * p) = raw;
  } else {
    uint2 raw;
    raw.x = floats_to_bf16x2(v[0], v[1]);
    raw.y = floats_to_bf16x2(v[2], v[3]);
    *reinterpret_cast<uint2 *>(row + 4 * p) = raw;
  }
}
// A loaded pack as it came from memory.  Loads fill a RawPack and nothing else, so that a thread
// can issue all the loads of a batch (or both loads of a row) without an instruction that
// depends on the data in between; `unpack` widens to fp32 registers at the point of use.
template <typename WT, int E>
struct RawPack;
template <int E>
struct RawPack<float, E> {
  float v[E];
};
template <>
struct RawPack<__nv_bfloat16, 8> {
  uint4 q;
};
template <>
struct RawPack<__nv_bfloat16, 4> {
  uint2 q;
};

template <int E>
__device__ __forceinline__ void unpack(const RawPack<float, E> &r, float (&v)[E]) {
#pragma unroll
  for (int i = 0; i < E; ++i) v[i] = r.v[i];
}
__device__ __forceinline__ void unpack(const RawPack<__nv_bfloat16, 8> &r, float (&v)[8]) {
  bf16x2_to_floats(r.q.x, v[0], v[1]);
  bf16x2_to_floats(r.q.y, v[2], v[3]);
  bf16x2_to_floats(r.q.z, v[4], v[5]);
  bf16x2_to_floats(r.q.w, v[6], v[7]);
}
__device__ __forceinline__ void unpack(const RawPack<__nv_bfloat16, 4> &r, float (&v)[4]) {
  bf16x2_to_floats(r.q.x, v[0], v[1]);
  bf16x2_to_floats(r.q.y, v[2], v[3]);
}

// fp32 values as a pack in storage form (bf16: to nearest even).
template <int E>
__device__ __forceinline__ void pack_raw(const float (&v)[E], RawPack<float, E> &r) {
#pragma unroll
  for (int i = 0; i < E; ++i) r.v[i] = v[i];
}
__device__ __forceinline__ void pack_raw(const float (&v)[8], RawPack<__nv_bfloat16, 8> &r) {
  r.q = make_uint4(floats_to_bf16x2(v[0], v[1]), floats_to_bf16x2(v[2], v[3]), floats_to_bf16x2(v[4], v[5]),
                   floats_to_bf16x2(v[6], v[7]));
}

// `at` points to the first element of the pack.  live == E: vector load; otherwise (the ragged
// last pack of a row) element by element, dead lanes read as 0.
template <int E>
__device__ __forceinline__ void ld_raw(const float *at, int live, RawPack<float, E> &r) {
  if (!access_ok(at, 4 * (size_t)live)) {  // debug build only: a skipped load reads as zeros
#pragma unroll
    for (int i = 0; i < E; ++i) r.v[i] = 0.f;
    return;
  }
  if (live == E) {
#pragma unroll
    for (int i = 0; i < E / 4; ++i) {
      const float4 t = *reinterpret_cast<const float4 *>(at + 4 * i);
      r.v[4 * i] = t.x; r.v[4 * i + 1] = t.y; r.v[4 * i + 2] = t.z; r.v[4 * i + 3] = t.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < E; ++i) r.v[i] = i < live ? at[i] : 0.f;
  }
}
__device__ __forceinline__ uint32_t ld_bf16_bits(const __nv_bfloat16 *at, int i, int live) {
  return i < live ? (uint32_t)*reinterpret_cast<const unsigned short *>(at + i) : 0u;
}
__device__ __forceinline__ void ld_raw(const __nv_bfloat16 *at, int live, RawPack<__nv_bfloat16, 8> &r) {
  if (!access_ok(at, 2 * (size_t)live)) {
    r.q = make_uint4(0u, 0u, 0u, 0u);
    return;
  }
  if (live == 8) {
    r.q = *reinterpret_cast<const uint4 *>(at);
  } else {
    r.q.x = ld_bf16_bits(at, 0, live) | (ld_bf16_bits(at, 1, live) << 16);
    r.q.y = ld_bf16_bits(at, 2, live) | (ld_bf16_bits(at, 3, live) << 16);
    r.q.z = ld_bf16_bits(at, 4, live) | (ld_bf16_bits(at, 5, live) << 16);
    r.q.w = ld_bf16_bits(at, 6, live) | (ld_bf16_bits(at, 7, live) << 16);
  }
}
__device__ __forceinline__ void ld_raw(const __nv_bfloat16 *at, int live, RawPack<__nv_bfloat16, 4> &r) {
  if (!access_ok(at, 2 * (size_t)live)) {
    r.q = make_uint2(0u, 0u);
    return;
  }
  if (live == 4) {
    r.q = *reinterpret_cast<const uint2 *>(at);
  } else {
    r.q.x = ld_bf16_bits(at, 0, live) | (ld_bf16_bits(at, 1, live) << 16);
    r.q.y = ld_bf16_bits(at, 2, live) | (ld_bf16_bits(at, 3, live) << 16);
  }
}
// The same pack back to memory as it is.
template <int E>
__device__ __forceinline__ void st_raw(float *at, int live, const RawPack<float, E> &r) {
  if (!access_ok(at, 4 * (size_t)live)) return;
  if (live == E) {
#pragma unroll
    for (int i = 0; i < E / 4; ++i)
      *reinterpret_cast<float4 *>(at + 4 * i) = make_float4(r.v[4 * i], r.v[4 * i + 1], r.v[4 * i + 2], r.v[4 * i + 3]);
  } else {
#pragma unroll
    for (int i = 0; i < E; ++i)
      if (i < live) at[i] = r.v[i];
  }
}
__device__ __forceinline__ void st_raw(__nv_bfloat16 *at, int live, const RawPack<__nv_bfloat16, 8> &r) {
  if (!access_ok(at, 2 * (size_t)live)) return;
  if (live == 8) {
    *reinterpret_cast<uint4 *>(at) = r.q;
  } else {
    const uint32_t words[4] = {r.q.x, r.q.y, r.q.z, r.q.w};
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (i < live) reinterpret_cast<unsigned short *>(at)[i] = (unsigned short)(words[i / 2] >> (16 * (i & 1)));
  }
}
template <typename WT, int E>
__device__ __forceinline__ void zero_raw(RawPack<WT, E> &r) {
  memset(&r, 0, sizeof(r));
}
template <typename T, int E>
__device__ __forceinline__ void st_pack_any(T *row, int64_t p, int live, const float (&v)[E]) {
  if (live == E) {
    st_pack<E>(row, p, v);
  } else {
#pragma unroll
    for (int i = 0; i < E; ++i)
      if (i < live) st_elem(row, E * p + i, v[i]);
  }
}
// Full packs (`live` is a compile-time E) of an arena whose rows start at multiples of 32 bytes: 8 fp32 values
// in one 32-byte store.  Two 16-byte stores of a warp cover half of each sector, and where L1 does not hold
// the line they reach L2 as two partial writes (30 % more write sectors in a batch that overwrites all
// devices).  Measured, us, two stores / one: resident batches, 16 devices, 2^24, one step 428 / 405 per round,
// 32 devices, 23.5 M 1602 / 1572; fused round, 8 devices, 11.2 M, one step 238.7 / 232.4; 16 devices, 2^25,
// one step 1300 / 1292.  A test of the address at each store cost what it gave (8 steps 578 -> 584 .. 588),
// hence the compile-time choice.  32-byte loads gain nothing (the line stays in L1 between the two halves)
// and cost bf16 rounds of 8 steps 2 %.
__device__ __forceinline__ void st_full(float *at, const float (&v)[8]) {
  if (!access_ok(at, 32)) return;
  asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(at), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]),
               "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]) : "memory");
}
template <int E>
struct FullPack {  // a number of live lanes that is E at compile time
  __device__ constexpr operator int() const { return E; }
};
template <typename T, int E>
__device__ __forceinline__ void st_pack_any(T *row, int64_t p, FullPack<E>, const float (&v)[E]) {
  if constexpr (sizeof(T) == 4 && E == 8)
    st_full(row + E * p, v);
  else
    st_pack<E>(row, p, v);
}
template <typename T>
__device__ __forceinline__ void st_raw(T *at, FullPack<8>, const RawPack<T, 8> &r) {
  if constexpr (sizeof(T) == 4)
    st_full(at, r.v);
  else
    st_raw(at, 8, r);
}
// Whether the fp32 rows behind w and m (their distance is a multiple of 32 bytes) start at multiples of 32.
template <typename WT, typename MT>
__device__ __forceinline__ bool rows_at_32(const WT *w, const MT *m) {
  const uintptr_t at = (sizeof(WT) == 4 ? (uintptr_t)w : 0) | (sizeof(MT) == 4 ? (uintptr_t)m : 0);
  return (at & 31) == 0;
}
// The value a parameter has once stored: itself for fp32, rounded to nearest even for bf16.
__device__ __forceinline__ float as_stored(float v, const float *) { return v; }
__device__ __forceinline__ float as_stored(float v, const __nv_bfloat16 *) {
  return __bfloat162float(__float2bfloat16_rn(v));
}
__device__ __forceinline__ int live_of(int64_t n_params, int64_t p, int E) {
  const int64_t left = n_params - (int64_t)E * p;
  return left >= E ? E : (left > 0 ? (int)left : 0);
}
template <int E>
__device__ __forceinline__ FullPack<E> live_of(std::true_type, int64_t, int64_t) {
  return {};
}
template <int E>
__device__ __forceinline__ int live_of(std::false_type, int64_t n_params, int64_t p) {
  return live_of(n_params, p, E);
}

// ------------------------------------------------------------------------------------------
// Uniform words -> standard normals (Box-Muller).  (x0, x1) -> (z0, z1):
//   u0 = (x0 + 0.5) 2^-32,  u1 = (x1 + 0.5) 2^-32,  r = sqrt(-2 ln u0),
//   z0 = r cos(2 pi u1),    z1 = r sin(2 pi u1).
// The angle is taken as a = u1 - [x1 >= 2^31] in (-1/2, 1/2), the same angle modulo a turn,
// by reading x1 as a signed integer: small angles keep their relative precision.
// ------------------------------------------------------------------------------------------

// Special-function-unit instructions in their flush-to-zero forms (no subnormal fix-up code; the
// arguments here are never subnormal).
__device__ __forceinline__ float sfu_sqrt(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float sfu_lg2(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float sfu_sin(float x) {
  float y;
  asm("sin.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float sfu_cos(float x) {
  float y;
  asm("cos.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// -2 ln(1 - t) by its series, for t = 1 - u0 = (~x0 + 0.5) 2^-32 < 2^-10, times `scale2`:
// 2t + t^2 + (2/3) t^3 (the next term, t^4/2, is below 2^-31 relative).  Only reached from a rarely
// taken branch (one combined test per step), so the common path pays a compare and an untaken
// branch for it; inlined there, because a real call inside the step loop makes the compiler shuffle
// the live registers around every call site (about one instruction per step on average).
__device__ __forceinline__ float r2_next_to_one(uint32_t x0, float scale2) {
  const float t = fmaf(__uint2float_rn(~x0), 0x1p-32f, 0x1p-33f);
  return scale2 * (t * fmaf(t, fmaf(t, 0.66666667f, 1.0f), 2.0f));
}

struct NormalsFast {
  // The four normals of standard deviation s of one Philox block (words x0 .. x3; pairs (x0, x1)
  // and (x2, x3)); the caller passes lg_scale = -2 ln2 s^2 and scale2 = s^2 so that the scaling
  // costs no instruction:
  //   r^2 = lg_scale * lg2(u0)            (u0 = (x0 + 0.5) 2^-32)
  //   theta = 2 pi a,  a = ((int)x1 + 0.5) 2^-32          (one fused multiply-add)
  // The fp32 arithmetic is written on packed pairs (sm_100's two-wide fp32 instructions: one issue
  // slot, two IEEE results): the block's two radii, its two angles, the two normals of a pair.
  // Next to u0 = 1 (x0 >= 2^32 - 2^22) lg2.approx only has an absolute error bound, so the exact
  // complement and a series take over.  Measured against a double-precision evaluation (s = 1):
  // max |dz| about 2e-6, mean 1.6e-7.
  static constexpr uint32_t kNearOne = 0xFFC00000u;
  // r^2 of both pairs, away from u0 = 1 (wrong by up to a few 1e-7 absolute next to it: see needs_series)
  static __device__ __forceinline__ float2 radius2_pair(uint32_t x0, uint32_t x2, float lg_scale) {
    const float2 u = __ffma2_rn(make_float2(__uint2float_rn(x0), __uint2float_rn(x2)),
                                make_float2(0x1p-32f, 0x1p-32f), make_float2(0x1p-33f, 0x1p-33f));
    return __fmul2_rn(make_float2(lg_scale, lg_scale), make_float2(sfu_lg2(u.x), sfu_lg2(u.y)));
  }
  static __device__ __forceinline__ bool needs_series(uint32_t x0) { return x0 >= kNearOne; }
  // theta of both pairs (words 1 and 3)
  static __device__ __forceinline__ float2 angle_pair(uint32_t x1, uint32_t x3) {
    return __ffma2_rn(make_float2(__int2float_rn((int)x1), __int2float_rn((int)x3)),
                      make_float2(1.4629180792671596e-9f, 1.4629180792671596e-9f),
                      make_float2(7.314590396335798e-10f, 7.314590396335798e-10f));
  }
  // (r cos theta, r sin theta)
  static __device__ __forceinline__ float2 finish_pair(float r2, float theta) {
    const float r = sfu_sqrt(r2);
    return __fmul2_rn(make_float2(r, r), make_float2(sfu_cos(theta), sfu_sin(theta)));
  }
  static __device__ __forceinline__ float4 block(uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3,
                                                 float lg_scale, float scale2) {
    float2 r2 = radius2_pair(x0, x2, lg_scale);
    if (needs_series(x0)) r2.x = r2_next_to_one(x0, scale2);
    if (needs_series(x2)) r2.y = r2_next_to_one(x2, scale2);
    const float2 theta = angle_pair(x1, x3);
    const float2 z01 = finish_pair(r2.x, theta.x), z23 = finish_pair(r2.y, theta.y);
    return make_float4(z01.x, z01.y, z23.x, z23.y);
  }
};

struct NormalsAccurate {
  // Full-precision fp32 library functions; the logarithm of u0 >= 1/2 is taken through the exact
  // complement 1 - u0 = (~x0 + 0.5) 2^-32 so that it keeps its relative accuracy next to 1.
  static __device__ __forceinline__ void pair(uint32_t x0, uint32_t x1, float lg_scale,
                                              float scale2, float &z0, float &z1) {
    (void)lg_scale;
    float neg_ln;
    if (x0 & 0x80000000u) {
      const float t = fmaf(__uint2float_rn(~x0), 0x1p-32f, 0x1p-33f);
      neg_ln = -log1pf(-t);
    } else {
      const float u0 = fmaf(__uint2float_rn(x0), 0x1p-32f, 0x1p-33f);
      neg_ln = -logf(u0);
    }
    const float a = fmaf(__int2float_rn((int)x1), 0x1p-32f, 0x1p-33f);
    const float r = sqrtf(2.0f * scale2 * neg_ln);
    float s, c;
    sincospif(2.0f * a, &s, &c);
    z0 = r * c;
    z1 = r * s;
  }
  static __device__ __forceinline__ float4 block(uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3,
                                                 float lg_scale, float scale2) {
    float4 z;
    pair(x0, x1, lg_scale, scale2, z.x, z.y);
    pair(x2, x3, lg_scale, scale2, z.z, z.w);
    return z;
  }
};

constexpr float kMinusTwoLn2 = -1.3862943611198906f;

// Unit normals of one Philox block.
template <typename Gen>
__device__ __forceinline__ float4 normals_of_block(uint32_t c0, uint32_t c1, uint32_t c2,
                                                   uint32_t c3, const PhiloxKeys &keys) {
  philox4x32_10(c0, c1, c2, c3, keys);
  return Gen::block(c0, c1, c2, c3, kMinusTwoLn2, 1.0f);
}

// ------------------------------------------------------------------------------------------
// K0: initial model.  Every row gets w_(0)[p] = init_std * z(seed; p), momentum 0; lanes beyond P
// (ragged group and row padding) are zeroed in both arenas.  One thread per column group of the
// padded row.
// ------------------------------------------------------------------------------------------
template <typename WT, typename MT>
__global__ void __launch_bounds__(kThreads)
k_init(WT *__restrict__ w, MT *__restrict__ m, int64_t stride, int64_t n_params, int n_devices,
       PhiloxKeys keys, float init_std) {
  const int64_t g = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  if (4 * g >= stride) return;
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (4 * g < n_params) {
    const float4 z = normals_of_block<NormalsAccurate>((uint32_t)g, 0u, 0u, kTagInit, keys);
    v.x = init_std * z.x;
    if (4 * g + 1 < n_params) v.y = init_std * z.y;
    if (4 * g + 2 < n_params) v.z = init_std * z.z;
    if (4 * g + 3 < n_params) v.w = init_std * z.w;
  }
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int i = 0; i < n_devices; ++i) {
    st_group(w + (int64_t)i * stride, g, v);
    st_group(m + (int64_t)i * stride, g, zero);
  }
}

// ------------------------------------------------------------------------------------------
// K1: batched local update (Eq. 3 / Algorithm 1) for a list of devices with per-device step
// counts, one launch.  A thread owns a pack of E columns (E/4 Philox blocks) and visits the listed
// rows one after the other: load w and m once, run that device's steps in registers (gradient
// from the counter-based generator), store once; other resident warps cover the load latency.
// The gradient noise grad_std * z is produced directly (the scale is
// folded into the constants of the radius), which differs from rounding z first by about one
// part in 10^7.
//
// The first Philox round of a gradient block multiplies the column-group index (fixed per thread)
// and the device id (fixed per row), so it is hoisted: the host folds the device product, the tag
// word and the first round keys into three words per row, the thread keeps the group product, and
// per step the round is two xors.  The host also guarantees that a row's step counter does not
// cross a multiple of 2^32 inside one launch (it splits the call), so the step index is one add.
// ------------------------------------------------------------------------------------------
struct RowStep {
  int64_t w_off;     // byte offset of the device's row in the parameter arena
  int64_t m_off;     // byte offset of the device's row in the momentum arena
  int32_t row;
  int32_t steps;
  uint32_t base_lo;  // low word of the device's step counter before this call
  uint32_t r1_c0;    // hi(M1 * device) ^ key_a[0]      (xor step index -> word 0)
  uint32_t r1_c1;    // lo(M1 * device)                                 (word 1)
  uint32_t r1_c2;    // (tag | step_hi) ^ key_b[0]   (xor hi(M0 * group) -> word 2)
};

struct LocalStepArgs {  // the host lists only devices that run at least one step
  int32_t n;
  RowStep r[kMaxDevices];
};

// Constants of the update, computed once on the host and read from the launch parameters:
// -lr, momentum, weight decay, -2 ln2 grad_std^2 and grad_std^2.
struct StepConsts {
  float neg_lr, mu, wd, lg_scale, scale2;
};

// The thread's share of the first Philox round: hi/lo of M0 * group for each of its NB groups.
template <int NB>
struct GroupProducts {
  uint32_t hi[NB], lo[NB];
  __device__ __forceinline__ explicit GroupProducts(int64_t pack) {
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const unsigned long long gp = (unsigned long long)kPhiloxM0 * (uint32_t)(pack * NB + b);
      hi[b] = (uint32_t)(gp >> 32);
      lo[b] = (uint32_t)gp;
    }
  }
};

// One SGD step of two parameters on packed pairs:
//   g = fma(wd, w, noise);  m = fma(mu, m, g);  w = fma(-lr, m, w)        (per lane, as in Eq. 3)
__device__ __forceinline__ void sgd_update_pair(float &w0, float &w1, float &m0, float &m1, float2 noise,
                                                float2 wd2, float2 mu2, float2 neg_lr2) {
  const float2 w2 = make_float2(w0, w1);
  const float2 g2 = __ffma2_rn(wd2, w2, noise);
  const float2 m2 = __ffma2_rn(mu2, make_float2(m0, m1), g2);
  const float2 w2n = __ffma2_rn(neg_lr2, m2, w2);
  w0 = w2n.x; w1 = w2n.y;
  m0 = m2.x; m1 = m2.y;
}

// The steps of one device on one pack.  Each step is written stage by stage over all NB Philox
// blocks of the pack - all generator rounds, then all radii, one combined test for the rare
// "u0 next to 1" case, then all angles, then the update - so that the independent chains sit in
// the same straight-line code and the hardware scheduler can interleave them.
// The fp32 arithmetic of a step is written on pairs (sm_100's two-wide fp32 instructions: one
// issue slot, two IEEE results, so every value is bit for bit what the scalar form gives): the two
// radii of a block, its two angles, the two normals of a Box-Muller pair and their two parameters.
// The launch is bound by the issue slot with several steps per device, and this takes 22 of 155
// warp instructions out of a step of an 8-parameter pack (measured: K1 -3 ... -4 %, fused round
// -4 ... -5 %).
// The gradient noise of step e for the NB column groups of a pack: nz[b] = grad_std * (z0, z1), (z2, z3).
// kVote: whether the rare logarithm series (about once in 250 steps of a pack) is asked for by the warp, so that the
// branch is taken by all lanes or by none and needs no convergence point; `lanes` are those of the warp that run the step.
// Measured, us, lane / warp: ResNet-18 size, 8 steps per device, fp32 local update 557.1 / 555.4, fused round 575.9 /
// 574.0; bf16 throughout, stochastic rounding, steps 1,1,2,2,4,4,8,8 2240 / 2236; batches of 16 devices with those
// steps 807.5 / 805.9; 32 devices, 2 M, bf16 parameters, one step 172 / 173.  Two builds for bf16 parameters with fp32
// momentum lose by it and ask each lane: the local update (8 steps 565 / 582, 2 steps 197 / 200.5), and the batch with a
// prefetch (32 devices, 2 M, 3 rounds 159 / 167; 16 devices, 1.5 M, 8 rounds 50.8 / 52.0), which spills more.
template <typename Gen, int NB, bool kVote = true>
__device__ __forceinline__ void step_noise(float2 (&nz)[NB][2], int e, const uint32_t (&c2_first)[NB],
                                           const GroupProducts<NB> &gp, const RowStep &rs, const PhiloxKeys &keys,
                                           const StepConsts &k, uint32_t lanes = 0xFFFFFFFFu) {
  const uint32_t c0_first = rs.r1_c0 ^ (rs.base_lo + (uint32_t)e);
  uint32_t x[NB][4];
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    x[b][0] = c0_first; x[b][1] = rs.r1_c1; x[b][2] = c2_first[b]; x[b][3] = gp.lo[b];
  }
#pragma unroll
  for (int r = 1; r < 10; ++r)
#pragma unroll
    for (int b = 0; b < NB; ++b) philox_round(x[b][0], x[b][1], x[b][2], x[b][3], keys.a[r], keys.b[r]);
  float2 r2[NB];  // squared radii of the block's two pairs
  uint32_t top = 0;
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    r2[b] = Gen::radius2_pair(x[b][0], x[b][2], k.lg_scale);
    top = max(top, max(x[b][0], x[b][2]));
  }
  bool series = Gen::needs_series(top);
  if (kVote) series = __any_sync(lanes, series);
  if (series) {
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      if (Gen::needs_series(x[b][0])) r2[b].x = r2_next_to_one(x[b][0], k.scale2);
      if (Gen::needs_series(x[b][2])) r2[b].y = r2_next_to_one(x[b][2], k.scale2);
    }
    if (kVote) __syncwarp(lanes);
  }
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const float2 theta = Gen::angle_pair(x[b][1], x[b][3]);
    nz[b][0] = Gen::finish_pair(r2[b].x, theta.x);
    nz[b][1] = Gen::finish_pair(r2[b].y, theta.y);
  }
}

template <int NB>
__device__ __forceinline__ void step_update(float (&w)[4 * NB], float (&m)[4 * NB], const float2 (&nz)[NB][2],
                                            const StepConsts &k) {
  const float2 wd2 = make_float2(k.wd, k.wd), mu2 = make_float2(k.mu, k.mu);
  const float2 neg_lr2 = make_float2(k.neg_lr, k.neg_lr);
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    sgd_update_pair(w[4 * b], w[4 * b + 1], m[4 * b], m[4 * b + 1], nz[b][0], wd2, mu2, neg_lr2);
    sgd_update_pair(w[4 * b + 2], w[4 * b + 3], m[4 * b + 2], m[4 * b + 3], nz[b][1], wd2, mu2, neg_lr2);
  }
}

// All steps of a row.  The loop is not unrolled: the copies
// would compute the step-independent products of the generator more than once (fused round 584 -> 578
// us at 8 steps per device, ResNet-18 size).
template <typename Gen, int NB, bool kVote = true>
__device__ __forceinline__ void sgd_steps(float (&w)[4 * NB], float (&m)[4 * NB],
                                          const GroupProducts<NB> &gp, const RowStep &rs,
                                          const PhiloxKeys &keys, const StepConsts &k, uint32_t lanes = 0xFFFFFFFFu) {
  uint32_t c2_first[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) c2_first[b] = gp.hi[b] ^ rs.r1_c2;
#pragma unroll 1
  for (int e = 0; e < rs.steps; ++e) {
    float2 nz[NB][2];
    step_noise<Gen, NB, kVote>(nz, e, c2_first, gp, rs, keys, k, lanes);
    step_update<NB>(w, m, nz, k);
  }
}

// ------------------------------------------------------------------------------------------
// Reduced-precision state (a workload variant outside the paper, which trains in fp32): the one
// rounding to bf16 at the end of a local-update call may be stochastic.  The 16 random bits are
// added to the fp32 bit pattern below the bf16 mantissa and the sum is truncated: a finite value
// moves to its neighbour of larger magnitude with probability (discarded bits) / 2^16, so the
// expectation is the value itself.  Infinities and NaNs are rounded to nearest even.
// The bits come from one Philox block per column group and call, counter
// (group, index of the call's last step, device, 'R' << 24 | index >> 32): element `lane` of the
// group takes the low half of word `lane` for its parameter and the high half for its momentum.
// The result is exactly representable in bf16, so the conversion at the store changes nothing.
// ------------------------------------------------------------------------------------------
// What bounds it is instructions: one more generator block per group (the first round's products are the
// gradients' own), then the values.  One test per pack finds out whether any of its values is not finite, where
// a test and a conversion per value stood, and what has been rounded here is not rounded again on its way to
// the aggregate.  Measured, us per round: 16 devices, 33.5 M parameters, steps 1,1,2,2,4,4,8,8, bf16
// throughout 2346 -> 2238; a batch of 8, 8 devices, 16.8 M, one step 301 -> 281.5.
__device__ __forceinline__ float bf16_stochastic(float v, uint32_t r16) {
  return __uint_as_float((__float_as_uint(v) + r16) & 0xFFFF0000u);
}
__device__ __forceinline__ float bf16_stochastic_any(float v, uint32_t r16) {
  if ((__float_as_uint(v) & 0x7F800000u) == 0x7F800000u) return __bfloat162float(__float2bfloat16_rn(v));
  return bf16_stochastic(v, r16);
}
// The larger magnitude, NaN if either is.
__device__ __forceinline__ float max_magnitude(float a, float b) {
  float m;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(fabsf(a)), "f"(fabsf(b)));
  return m;
}

// kTogether: the test is the warp's, for rows that go to tensor memory afterwards, whose instructions want all lanes
// together.  (Elsewhere a pack's own is the faster one: the round above 2237 us, with the warp's 2255; 32 devices, 2 M 200 /
// 203.  Rows on the SM: 16 devices, 4.2 M, one step 147.2 / 146.0.)
template <typename MT, bool kTogether, int NB>
__device__ __forceinline__ void round_stochastic(float (&w)[4 * NB], float (&m)[4 * NB], const GroupProducts<NB> &gp,
                                                 const RowStep &rs, const PhiloxKeys &keys) {
  constexpr int E = 4 * NB;
  uint32_t x[NB][4];
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    x[b][0] = rs.r1_c0 ^ (rs.base_lo + (uint32_t)rs.steps - 1u);
    x[b][1] = rs.r1_c1;
    x[b][2] = gp.hi[b] ^ rs.r1_c2 ^ (kTagGrad ^ kTagRound);
    x[b][3] = gp.lo[b];
  }
#pragma unroll
  for (int r = 1; r < 10; ++r)
#pragma unroll
    for (int b = 0; b < NB; ++b) philox_round(x[b][0], x[b][1], x[b][2], x[b][3], keys.a[r], keys.b[r]);
  float largest = max_magnitude(w[0], w[1]);
#pragma unroll
  for (int i = 2; i < E; ++i) largest = max_magnitude(largest, w[i]);
  if (sizeof(MT) == 2) {
#pragma unroll
    for (int i = 0; i < E; ++i) largest = max_magnitude(largest, m[i]);
  }
  bool finite = largest < __uint_as_float(0x7F800000u);
  if (kTogether) finite = __all_sync(0xFFFFFFFFu, finite);
  if (finite) {
#pragma unroll
    for (int i = 0; i < E; ++i) {
      w[i] = bf16_stochastic(w[i], x[i / 4][i % 4] & 0xFFFFu);
      if (sizeof(MT) == 2) m[i] = bf16_stochastic(m[i], x[i / 4][i % 4] >> 16);
    }
  } else {
#pragma unroll
    for (int i = 0; i < E; ++i) {
      w[i] = bf16_stochastic_any(w[i], x[i / 4][i % 4] & 0xFFFFu);
      if (sizeof(MT) == 2) m[i] = bf16_stochastic_any(m[i], x[i / 4][i % 4] >> 16);
    }
    if (kTogether) __syncwarp();
  }
}

// Row addressing: the host passes each row's byte offset, the thread adds the byte offset of its
// pack once, so a row access costs one 64-bit add.
template <typename WT>
__device__ __forceinline__ WT *at_row(char *pack_in_row0, int64_t row_off) {
  return reinterpret_cast<WT *>(pack_in_row0 + row_off);
}

// WT / MT: storage types of the parameters and of the momentum (bf16 momentum only with bf16
// parameters); RM = 1: the bf16 stores of this call are rounded stochastically.
template <typename WT, typename MT, typename Gen, int E, int RM>
__global__ void __launch_bounds__(kThreads)
k_local_step(WT *__restrict__ w, MT *__restrict__ m, int64_t n_params, LocalStepArgs a,
             PhiloxKeys keys, StepConsts k) {
  constexpr bool kVote = !(sizeof(WT) == 2 && sizeof(MT) == 4 && RM == 0);  // (measured at step_noise)
  const int64_t p = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  // The body is compiled twice: for blocks whose packs are all full (`live` is then the constant
  // E and every ragged-tail test in the loads and stores folds away: 2-3 % fewer instructions per
  // row, and 32-byte stores) and for the one block that holds the end of the vector, or all blocks of an arena
  // whose rows do not start at multiples of 32 bytes.
  auto run = [&](auto all_full) {
    const auto live = live_of<E>(all_full, n_params, p);
    // Lanes beyond the end of the vector are done: running along - a warp of them, or next to live ones, which then went
    // through the loads and stores of both kinds - they made the block with the end the last one to finish (4 steps per
    // device: 6 devices of 300,007 bf16 parameters 11.8 us without them, 13.3 with; 32 of 200,000 in fp32 44.5 / 49.0).
    uint32_t lanes = 0xFFFFFFFFu;
    if constexpr (!decltype(all_full)::value) {
      lanes = __ballot_sync(0xFFFFFFFFu, live > 0);
      if (live == 0) return;
    }
    const GroupProducts<E / 4> gp(p);
    char *wp = reinterpret_cast<char *>(w) + p * (int64_t)(E * sizeof(WT));
    char *mp = reinterpret_cast<char *>(m) + p * (int64_t)(E * sizeof(MT));

    auto load = [&](int j, RawPack<WT, E> &rw, RawPack<MT, E> &rm) {
      ld_raw(at_row<WT>(wp, a.r[j].w_off), live, rw);
      ld_raw(at_row<MT>(mp, a.r[j].m_off), live, rm);
    };
    auto body = [&](int j, float (&wv)[E], float (&mv)[E]) {
      sgd_steps<Gen, E / 4, kVote>(wv, mv, gp, a.r[j], keys, k, lanes);
      if constexpr (RM == 1) round_stochastic<MT, false>(wv, mv, gp, a.r[j], keys);
      st_pack_any(at_row<WT>(wp, a.r[j].w_off), 0, live, wv);
      st_pack_any(at_row<MT>(mp, a.r[j].m_off), 0, live, mv);
    };
    // fp32 values are updated in the registers they were loaded into; bf16 ones are widened first
    auto visit = [&](int j, RawPack<WT, E> &rw, RawPack<MT, E> &rm) {
      if constexpr (sizeof(WT) == 4) {
        body(j, rw.v, rm.v);
      } else if constexpr (sizeof(MT) == 4) {
        float wv[E];
        unpack(rw, wv);
        body(j, wv, rm.v);
      } else {
        float wv[E], mv[E];
        unpack(rw, wv);
        unpack(rm, mv);
        body(j, wv, mv);
      }
    };
    // No prefetch of the next row: the registers it would take cost a resident block, and four
    // blocks per SM hide the row loads better than three blocks with a prefetch (measured).
    // Grid: x = chunks of kThreads packs; y = 1: the block walks over all listed rows (every thread
    // mixes light and heavy rows, so memory-bound and arithmetic-bound phases overlap), or
    // y = number of rows: one row per block (eight times more, shorter blocks: no partial last
    // wave, which is worth 5-7 % when every row is memory-bound).  The host chooses.
    RawPack<WT, E> rw;
    RawPack<MT, E> rm;
    const int j_begin = gridDim.y > 1 ? (int)blockIdx.y : 0;
    const int j_end = gridDim.y > 1 ? j_begin + 1 : a.n;
    for (int j = j_begin; j < j_end; ++j) {
      load(j, rw, rm);
      visit(j, rw, rm);
    }
  };
  if (((int64_t)blockIdx.x + 1) * kThreads * E <= n_params && rows_at_32(w, m))
    run(std::true_type{});
  else
    run(std::false_type{});
}

// ------------------------------------------------------------------------------------------
// K2: fused weighted combination of `nr` rows written to `nw` rows in the same pass.
//   partial aggregation (Eq. 5): read list = write list = the selected devices, weights a_j;
//   global synchronisation (Algorithm 1): read list = {source}, weight 1, write list = receivers.
//   acc = a_0 * w[rd_0];  acc = fma(a_j, w[rd_j], acc) for j = 1 .. nr-1, in list order.
// A thread owns U 16-byte packs.  KR > 0: compile-time read count; KR == 0: any read count.  The
// row loads of a pack are issued in batches of B rows (B * E values in registers) before the
// batch's multiply-adds; U packs per thread keep enough bytes in flight when the list is short.
// ------------------------------------------------------------------------------------------
struct CombineArgs {
  int32_t nr;
  int32_t nw;
  int32_t rd[kMaxDevices];
  float a[kMaxDevices];
  int32_t wr[kMaxDevices];
};

template <typename WT, int KR, int E>
__device__ __forceinline__ void combine_pack(const WT *__restrict__ w, int64_t stride,
                                             const CombineArgs &c, int64_t p, int live,
                                             float (&acc)[E]) {
  constexpr int B = KR > 0 ? (KR <= 16 ? KR : 16) : 8;  // rows per batch: at most 16 x 16 bytes in registers
  const int nr = KR > 0 ? KR : c.nr;
#pragma unroll
  for (int i = 0; i < E; ++i) acc[i] = 0.f;
#pragma unroll
  for (int base = 0; base < (KR > 0 ? KR : kMaxDevices); base += B) {
    if (base >= nr) break;
    RawPack<WT, E> raw[B];
#pragma unroll
    for (int j = 0; j < B; ++j)
      if (base + j < nr) ld_raw(w + (int64_t)c.rd[base + j] * stride + (int64_t)E * p, live, raw[j]);
#pragma unroll
    for (int j = 0; j < B; ++j) {
      if (base + j < nr) {
        const float aj = c.a[base + j];
        float v[E];
        unpack(raw[j], v);
        if (base + j == 0) {
#pragma unroll
          for (int i = 0; i < E; ++i) acc[i] = __fmul_rn(aj, v[i]);
        } else {
#pragma unroll
          for (int i = 0; i < E; ++i) acc[i] = fmaf(aj, v[i], acc[i]);
        }
      }
    }
  }
}

template <typename WT, int KR, int U>
__global__ void __launch_bounds__(kThreads)
k_combine(WT *__restrict__ w, int64_t stride, int64_t n_params, CombineArgs c) {
  constexpr int E = Pack16<WT>::E;
  // Blocks walk the vector from its END to its start: the local update before it in a round walks
  // it from the start, so what that kernel left in the 126 MB L2 - the end of every row - is read
  // first.  Measured inside a round on the ResNet-18-sized workload (k = 4): 159 of the 179 MB of
  // reads come from DRAM instead of all of them, 61 -> 57 us.
  const int64_t chunk = (int64_t)(gridDim.x - 1 - blockIdx.x);
  const int64_t p0 = chunk * (kThreads * U) + threadIdx.x;
  // Fast path (all but the last chunk of a launch): every pack of the block is full, so the
  // U * KR row loads of a thread are straight-line code and all in flight together.
  const bool block_full = ((chunk + 1) * (kThreads * U)) * E <= n_params;
  if (KR > 0 && KR * U <= 16 && block_full) {
    constexpr int KRc = KR > 0 ? KR : 1;
    RawPack<WT, E> raw[U][KRc];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int j = 0; j < KRc; ++j)
        ld_raw(w + (int64_t)c.rd[j] * stride + (int64_t)E * (p0 + (int64_t)u * kThreads), E, raw[u][j]);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      float acc[E], v[E];
      unpack(raw[u][0], v);
#pragma unroll
      for (int i = 0; i < E; ++i) acc[i] = __fmul_rn(c.a[0], v[i]);
#pragma unroll
      for (int j = 1; j < KRc; ++j) {
        unpack(raw[u][j], v);
#pragma unroll
        for (int i = 0; i < E; ++i) acc[i] = fmaf(c.a[j], v[i], acc[i]);
      }
      for (int j = 0; j < c.nw; ++j)
        st_pack<E>(w + (int64_t)c.wr[j] * stride, p0 + (int64_t)u * kThreads, acc);
    }
    return;
  }
  float acc[U][E];
  int live[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int64_t p = p0 + (int64_t)u * kThreads;
    live[u] = live_of(n_params, p, E);
    if (live[u] > 0) combine_pack<WT, KR, E>(w, stride, c, p, live[u], acc[u]);
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int64_t p = p0 + (int64_t)u * kThreads;
    if (live[u] > 0)
      for (int j = 0; j < c.nw; ++j) st_pack_any(w + (int64_t)c.wr[j] * stride, p, live[u], acc[u]);
  }
}

// ------------------------------------------------------------------------------------------
// Integration of a received model (Section "Model aggregation and fault-tolerant": an unselected
// device folds the received parameters into its own; read here as a convex combination, beside the
// overwrite that k_combine provides):
//   w[dst_j] = fma(beta, w[src], (1 - beta) * w[dst_j])   for every receiver j,
// the product rounded to fp32 before the fused multiply-add.  A thread owns U 16-byte packs; per
// pack the sender's values are loaded once and the receivers' rows are loaded in batches of 8
// before the batch's arithmetic and stores.  1 + n reads and n writes per element.
// ------------------------------------------------------------------------------------------
struct MixArgs {
  int32_t n;    // receivers
  int32_t src;  // sender
  float beta, one_minus_beta;
  int32_t dst[kMaxDevices];
};

template <typename WT, int U>
__global__ void __launch_bounds__(kThreads)
k_integrate(WT *__restrict__ w, int64_t stride, int64_t n_params, MixArgs a) {
  constexpr int E = Pack16<WT>::E;
  constexpr int B = 8;
  const int64_t p0 = (int64_t)blockIdx.x * (kThreads * U) + threadIdx.x;
  int live[U];
  RawPack<WT, E> from[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int64_t p = p0 + (int64_t)u * kThreads;
    live[u] = live_of(n_params, p, E);
    if (live[u] > 0) ld_raw(w + (int64_t)a.src * stride + (int64_t)E * p, live[u], from[u]);
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    if (live[u] == 0) continue;
    const int64_t p = p0 + (int64_t)u * kThreads;
    float s[E];
    unpack(from[u], s);
    for (int base = 0; base < a.n; base += B) {
      RawPack<WT, E> raw[B];
#pragma unroll
      for (int j = 0; j < B; ++j)
        if (base + j < a.n) ld_raw(w + (int64_t)a.dst[base + j] * stride + (int64_t)E * p, live[u], raw[j]);
#pragma unroll
      for (int j = 0; j < B; ++j) {
        if (base + j < a.n) {
          float v[E];
          unpack(raw[j], v);
#pragma unroll
          for (int i = 0; i < E; ++i) v[i] = fmaf(a.beta, s[i], __fmul_rn(a.one_minus_beta, v[i]));
          st_pack_any(w + (int64_t)a.dst[base + j] * stride, p, live[u], v);
        }
      }
    }
  }
}

// ------------------------------------------------------------------------------------------
// Deterministic reductions shared by the statistics kernel and the fused round kernel.
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
  return v;
}

// The finish's sums: emit(t, sum of src[t][0 .. n_src)) for every t < n_vals, by one block, in a fixed order
// (a warp per value, lanes strided, then the butterfly).  Often only this block is still running, so
// what counts is latency: a warp takes 2 values at a time and has up to 8 loads in flight.  Measured
// against one load in flight (and, in a launch of 8 rounds, one finish per round): statistics kernel 52.1
// -> 49.2 us (32 devices, 2 M parameters), a single fused round of 32 devices 189 -> 184 us, 8 rounds in
// one launch 6.8 -> 5.2 us per round (4 devices, 100,000 parameters) and 162 -> 147 us (8 devices, 11 M).
template <typename Emit>
__device__ __forceinline__ void sum_partials(const double *__restrict__ src, int64_t stride, int n_vals, int n_src,
                                             Emit emit) {
  constexpr int kVals = 2, kLoads = 4;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
#pragma unroll 1
  for (int t0 = warp * kVals; t0 < n_vals; t0 += n_warps * kVals) {
    double s[kVals] = {};
#pragma unroll 1
    for (int l0 = lane; l0 < n_src; l0 += 32 * kLoads) {
      double v[kVals][kLoads];
#pragma unroll
      for (int i = 0; i < kVals; ++i)
#pragma unroll
        for (int q = 0; q < kLoads; ++q) {
          const int l = l0 + 32 * q;
          v[i][q] = t0 + i < n_vals && l < n_src ? __ldcg(src + (int64_t)(t0 + i) * stride + l) : 0.0;
        }
#pragma unroll
      for (int i = 0; i < kVals; ++i)
#pragma unroll
        for (int q = 0; q < kLoads; ++q) s[i] += v[i][q];
    }
#pragma unroll
    for (int i = 0; i < kVals; ++i) s[i] = warp_sum(s[i]);
#pragma unroll
    for (int i = 0; i < kVals; ++i)
      if (lane == 0 && t0 + i < n_vals) emit(t0 + i, s[i]);
  }
}

// Whether this block draws the last of n tickets; what it wrote before is visible to the block that does.
__device__ __forceinline__ bool is_last_block(unsigned int *__restrict__ ticket, unsigned int n, bool *s_last) {
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) *s_last = (atomicAdd(ticket, 1u) == n - 1u);
  __syncthreads();
  if (!*s_last) return false;
  __threadfence();
  return true;
}

// Last-block finish: the block that draws the last ticket sums partials[t][0 .. n_src) for every
// t < n_vals in a fixed order (a warp per value, lanes strided, then the butterfly), hands the
// sums to `emit`, and resets the ticket.  Returns without waiting for anyone.
template <typename Emit>
__device__ __forceinline__ void finish_by_last_block(const double *__restrict__ partials,
                                                     int n_vals, int n_src,
                                                     unsigned int *__restrict__ ticket,
                                                     bool *s_last, Emit emit) {
  if (!is_last_block(ticket, gridDim.x, s_last)) return;
  sum_partials(partials, n_src, n_vals, n_src, emit);
  if (threadIdx.x == 0) *ticket = 0u;
}

// Finish for grids of many blocks (the fused round), in two levels.  Blocks are grouped in runs of
// kFinishGroup consecutive block indices.  The block that draws a group's last ticket sums that
// group's partials[t][first block of the group ...] in block order -> group_partials[t][group]
// and draws the launch's ticket; the block that draws the last of those sums the group sums in
// group order and hands them to `emit`.  Each of the two sums has a fixed order that does not
// depend on which block happens to compute it, so the result is reproducible; no block waits for
// another; all tickets are back at zero when the launch ends.
constexpr int kFinishGroup = 128;

// Both levels by one block, for up to 4 groups, in the same order: the order must not depend on which of the two a
// launch takes, since that follows from its number of rounds and a batch leaves the statistics that single rounds do.
// A warp takes two values of two groups at a time, all 16 loads of a lane in flight.  The butterflies over the lanes are
// folded into one: lanes 0 .. 15 go on with the first value and 16 .. 31 with the second, the odd eights with the
// second group, and every sum is that of the whole butterfly (lane l has what lane l of it would have).  The group sums
// G0 .. G3 then meet as in the second level: (G0 + G2) + (G1 + G3).
template <typename Emit>
__device__ __forceinline__ void sum_up_to_four_groups(const double *__restrict__ partials, int n_vals, int n_blocks, Emit emit) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
  const bool second = (lane & 16) != 0, odd = (lane & 8) != 0;
#pragma unroll 1
  for (int t0 = warp * 2; t0 < n_vals; t0 += n_warps * 2) {
    double sum = 0.0;
#pragma unroll 1
    for (int first = 0; first < n_blocks; first += 2 * kFinishGroup) {
      double v[2][2][4], p[2][2] = {};
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int g = 0; g < 2; ++g)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int l = first + g * kFinishGroup + 32 * q + lane;
            v[i][g][q] = t0 + i < n_vals && l < n_blocks ? __ldcg(partials + (int64_t)(t0 + i) * n_blocks + l) : 0.0;
          }
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int g = 0; g < 2; ++g)
#pragma unroll
          for (int q = 0; q < 4; ++q) p[i][g] += v[i][g][q];
      double d[2];
#pragma unroll
      for (int g = 0; g < 2; ++g)
        d[g] = (second ? p[1][g] : p[0][g]) + __shfl_xor_sync(0xFFFFFFFFu, second ? p[0][g] : p[1][g], 16);
      double s = (odd ? d[1] : d[0]) + __shfl_xor_sync(0xFFFFFFFFu, odd ? d[0] : d[1], 8);
#pragma unroll
      for (int off = 4; off > 0; off >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
      sum += s;
    }
    sum += __shfl_xor_sync(0xFFFFFFFFu, sum, 8);
    const int t = t0 + (lane >> 4);
    if ((lane & 15) == 0 && t < n_vals) emit(t, sum);
  }
}

// The same for up to kPartSums sums that are in kParts parts each, which are added first: part i of sum s is number
// s * kParts + i of the n_src, and at partials[value][i][s].  All loads of a lane in flight, without a condition (one that
// waits for the load before it costs as much again); what lies beyond the end is left out afterwards.
constexpr int kPartSums = 160;
template <int kParts, typename Emit>
__device__ __forceinline__ void sum_parts(const double *__restrict__ partials, int n_vals, int n_src, int n_sums, Emit emit) {
  constexpr int kVals = kParts == 2 ? 2 : 1, kLoads = kPartSums / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
  const bool upper = (lane & 16) != 0;
#pragma unroll 1
  for (int t0 = warp * kVals; t0 < n_vals; t0 += n_warps * kVals) {
    const double *mine = partials + t0 * kParts * n_sums;
    double v[kVals][kParts][kLoads];
#pragma unroll
    for (int q = 0; q < kLoads; ++q) {
      const double *at = mine + min(32 * q + lane, n_sums - 1);
#pragma unroll
      for (int i = 0; i < kVals * kParts; ++i, at += n_sums) v[i / kParts][i % kParts][q] = __ldcg(at);
    }
#pragma unroll
    for (int k = 0; k < kVals; ++k) {
      double p[2] = {};
#pragma unroll
      for (int q = 0; q < kLoads; ++q) {
        double sum = 0.0;
#pragma unroll
        for (int i = 0; i < kParts; ++i) sum += (32 * q + lane) * kParts + i < n_src ? v[k][i][q] : 0.0;
        p[32 * q / kFinishGroup] += sum;
      }
      double s = (upper ? p[1] : p[0]) + __shfl_xor_sync(0xFFFFFFFFu, upper ? p[0] : p[1], 16);
#pragma unroll
      for (int off = 8; off > 0; off >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
      s += __shfl_xor_sync(0xFFFFFFFFu, s, 16);
      if (lane == 0) emit(t0 + k, s);
    }
  }
}

// Launches of few blocks are finished by one block, the last one: a second level's fence, ticket and loads come after
// the last block's work.  One block's warps add two values at a time (a turn) and two groups of each at a time, one wait
// for L2 after the other: up to 2 groups that costs less than the second level, up to 4 with four turns at most, and
// beyond that it grows with the blocks.  Measured, us per launch of one round, two levels / one (values x blocks): 4
// devices 8 x 196 8.8 / 6.8, 8 x 512 13.5 / 12.2; one device 2 x 512 7.7 / 6.3; 16 devices 32 x 256 26.2 / 23.7; 32
// devices 64 x 256 58.5 / 54.4, 64 x 512 97.1 / 95.9; 8 rounds in one launch, 512 x 147 53.2 / 48.7 per round.  Beyond the
// lines (one level as one sequence of all the blocks' sums): one device 2 x 1024 11.1 / 11.7, 2 x 8192 57.6 / 80.1; 2 devices
// 4 x 4096 50.1 / 62.7; 8 devices 16 x 1024 48.0 / 49.2.
template <typename Emit>
__device__ __forceinline__ void finish_by_groups(const double *__restrict__ partials,
                                                 double *__restrict__ group_partials, int n_vals,
                                                 unsigned int *__restrict__ group_tickets,
                                                 unsigned int *__restrict__ ticket, bool *s_last,
                                                 Emit emit) {
  const int n_blocks = (int)gridDim.x;
  const int four_turns = (int)blockDim.x / 4;  // values: 4 x 2 per warp
  const bool one_level = n_blocks <= 2 * kFinishGroup || (n_blocks <= 4 * kFinishGroup && n_vals <= four_turns);
  const int n_groups = one_level ? 1 : (n_blocks + kFinishGroup - 1) / kFinishGroup;
  const int g = one_level ? 0 : (int)blockIdx.x / kFinishGroup;
  const int g_first = g * kFinishGroup;
  const int g_size = one_level ? n_blocks : min(kFinishGroup, n_blocks - g_first);
  if (!is_last_block(group_tickets + g, (unsigned)g_size, s_last)) return;
  if (one_level) {
    sum_up_to_four_groups(partials, n_vals, n_blocks, emit);
    if (threadIdx.x == 0) group_tickets[0] = 0u;
    return;
  }
  sum_partials(partials + g_first, n_blocks, n_vals, g_size, [&](int t, double s) {
    if (access_ok(group_partials + (int64_t)t * n_groups + g, 8)) group_partials[(int64_t)t * n_groups + g] = s;
  });
  if (threadIdx.x == 0) group_tickets[g] = 0u;
  if (!is_last_block(ticket, (unsigned)n_groups, s_last)) return;
  sum_partials(group_partials, n_groups, n_vals, n_groups, emit);
  if (threadIdx.x == 0) *ticket = 0u;
}

// ------------------------------------------------------------------------------------------
// K3: per-replica squared norm and squared distance to a reference replica.
// Block b works on row b % N and on the chunks (b / N), (b / N) + lanes, ...; a chunk is
// kThreads * U 16-byte packs.  Blocks that are neighbours in launch order work on the same chunk
// of different rows at about the same time, so the reference chunk is fetched from HBM once and
// found in L2 by the others: HBM traffic stays N * P elements.
// Per thread: fp32 sums over the elements of a chunk in a fixed order, accumulated in fp64 across
// chunks; butterfly over the warp and a fixed-order sum over the warps (fp64) give
// partials[which * N + row][lane].  The last-ticket block sums them -> out[2N] (norm2 then div2).
// No block waits for another; fixed grid and fixed orders make the result reproducible.
// ------------------------------------------------------------------------------------------
template <typename WT, int U>
__global__ void __launch_bounds__(kThreads)
k_stats(const WT *__restrict__ w, int64_t stride, int64_t n_params, int n_devices, int ref,
        int lanes, double *__restrict__ partials, unsigned int *__restrict__ ticket,
        float *__restrict__ out) {
  constexpr int kWarps = kThreads / 32;
  constexpr int E = Pack16<WT>::E;
  __shared__ double s_part[2][kWarps];
  __shared__ bool s_last;
  const int row = blockIdx.x % n_devices;
  const int my_lane = blockIdx.x / n_devices;
  const int64_t n_packs = (n_params + E - 1) / E;
  const int64_t per_chunk = (int64_t)kThreads * U;
  const int64_t n_chunks = (n_packs + per_chunk - 1) / per_chunk;
  const WT *my_row = w + (int64_t)row * stride;
  const WT *ref_row = w + (int64_t)ref * stride;

  double n2 = 0.0, d2 = 0.0;
  for (int64_t chunk = my_lane; chunk < n_chunks; chunk += lanes) {
    const int64_t p0 = chunk * per_chunk + threadIdx.x;
    RawPack<WT, E> rv[U], rr[U];
    if ((chunk + 1) * per_chunk * E <= n_params) {  // every pack of the chunk is full: no branches
#pragma unroll
      for (int u = 0; u < U; ++u) {
        ld_raw(my_row + (int64_t)E * (p0 + (int64_t)u * kThreads), E, rv[u]);
        ld_raw(ref_row + (int64_t)E * (p0 + (int64_t)u * kThreads), E, rr[u]);
      }
    } else {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int64_t p = p0 + (int64_t)u * kThreads;
        const int live = live_of(n_params, p, E);
        if (live > 0) {
          ld_raw(my_row + (int64_t)E * p, live, rv[u]);
          ld_raw(ref_row + (int64_t)E * p, live, rr[u]);
        } else {
          zero_raw(rv[u]);
          zero_raw(rr[u]);
        }
      }
    }
    float a = 0.f, b = 0.f;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      float v[E], r[E];
      unpack(rv[u], v);
      unpack(rr[u], r);
#pragma unroll
      for (int i = 0; i < E; ++i) {
        const float d = v[i] - r[i];
        a = fmaf(v[i], v[i], a);
        b = fmaf(d, d, b);
      }
    }
    n2 += (double)a;
    d2 += (double)b;
  }
  n2 = warp_sum(n2);
  d2 = warp_sum(d2);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) {
    s_part[0][warp] = n2;
    s_part[1][warp] = d2;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    double s = 0.0;
    for (int wi = 0; wi < kWarps; ++wi) s += s_part[threadIdx.x][wi];
    double *slot = partials + ((int64_t)threadIdx.x * n_devices + row) * lanes + my_lane;
    if (access_ok(slot, 8)) *slot = s;
  }
  finish_by_last_block(partials, 2 * n_devices, lanes, ticket, &s_last,
                       [&](int t, double sum) {
                         if (access_ok(out + t, 4)) out[t] = (float)sum;
                       });
}

// ------------------------------------------------------------------------------------------
// Fused round: local update of every device, partial aggregation with write-back (optionally
// sent to every device: global synchronisation) and the statistics, in ONE pass over the arena.
// Selection only needs the versions, which the host knows before the steps run, so the selected
// set is an input.  Per pack a thread visits the rows in the order "selected devices in draw
// order, then the others": it runs each row's steps in registers exactly as K1 does, folds the
// selected rows into the aggregate in draw order exactly as K2 does (acc = a_0 w_0, then fma),
// writes the aggregate to the selected rows when the last of them is done, and for every row adds
// the squares of what the row now holds, and of its distance to the aggregate, to the row's sums.
// Parameters and momentum come out bit-identical to K1 followed by K2 (and the broadcast); the
// aggregate is never re-read from memory, so a round moves 16 bytes per (device, parameter)
// instead of 20 + 8k/N.
//
// Grid: one block per chunk of kThreads packs, up to a cap beyond which the blocks stride over
// the chunks; the hardware block scheduler then balances the SMs (a one-wave persistent grid ends
// with a partly filled last pass and keeps all blocks in the same phase of their rows: measured
// 7-15 % slower with several steps per device).  The chunk loop's trip count depends on the block
// index only, so control flow and every row descriptor read inside it are uniform across the
// block - with a per-thread loop bound the compiler re-read the descriptors through indexed
// constant loads in every step (+7 instructions per step).  Lanes beyond the end of the vector
// (live = 0) take part in everything: their loads return zeros, their stores store nothing, and
// what they compute is zeroed before it is summed.
// Row sums: one shuffle per row and pack, then a shared-memory slot owned by the thread (fp32); at
// the end of a chunk's round, per row, a fixed-order sum over the warps and a butterfly over each
// half-warp (fp64), added to the block's sums of that round; at the end of the block
// partials[round][value][block] and one last-ticket finish.  Deterministic.
// Dynamic shared memory: n * kThreads floats.  64 registers: four resident blocks per SM.
// NR > 1: the launch takes a batch of up to NR consecutive rounds.  A block carries its chunk
// through all of them before it moves on (chunk loop outside, round loop inside), so from the
// second round on the rows come from L2 and not from HBM, and every round still leaves its own
// statistics.  Results are those of the rounds launched one by one, bit for bit.
// E = 4 (fp32 only): packs of 4 columns, one Philox block per thread.  A block then holds half
// the rows at a time, which keeps the rows of all resident blocks within the L2 for up to about
// 20 devices: the form batches of one-step rounds take (the host decides).  Statistics are then
// folded over chunks of 1024 columns: equal to the other forms to rounding, not bit for bit.
// PF = true is a second build that issues the next row's loads before the current row's steps
// (80 registers, three resident blocks).  With bf16 parameters a row is 48 bytes per thread or
// less, and when every device runs one or two steps the launch is bound by how many bytes are in
// flight: the prefetch is worth 6-8 % there (and costs 1-3 % with more steps, and 0-13 % with fp32
// parameters at any step count), so the host takes it for exactly that case.
// ------------------------------------------------------------------------------------------
struct RoundArgs {
  int32_t n;          // rows visited = all N devices: [0, k) selected in draw order, then the rest
  int32_t k;          // number of selected devices, 1 <= k <= n
  int32_t write_all;  // global synchronisation: 0 none, 1 every other device receives the aggregate
                      // (overwrite), 2 every other device mixes it into its own model
  float beta, one_minus_beta;  // weights of the mix (write_all = 2), as in k_integrate
  float a[kMaxDevices];  // aggregation weights of the selected devices
  RowStep r[kMaxDevices];
};

// Adds a thread's (sum of squares, sum of squared distances) for one row to the block's
// accumulators.  One shuffle folds lane l and lane l ^ 16 so that the lower half-warp carries the
// first value and the upper half the second; each thread then owns ONE fp32 slot per row,
// s_acc[visit index][thread], which it alone updates (no atomics, fixed order).
__device__ __forceinline__ void add_row_sums(float *s_acc, int j, float n2, float d2, int lane) {
  const bool upper = (lane & 16) != 0;
  const float keep = upper ? d2 : n2;
  const float give = upper ? n2 : d2;
  float *slot = s_acc + j * kThreads + threadIdx.x;
  *slot += keep + __shfl_xor_sync(0xFFFFFFFFu, give, 16);
}

constexpr int kRoundBlocksPerSM = 4;

// A batch of consecutive rounds for one launch.  Every operation of a round is elementwise in the
// parameter index and the selections are known to the host beforehand, so a thread can take its
// pack through several rounds back to back: what it wrote in one round it reads back in the next
// (the same thread, the same addresses, program order), while the lines are still in L2.
template <int NR>
struct RoundBatch {
  int32_t n_rounds;  // 1 <= n_rounds <= NR
  RoundArgs round[NR];
};
constexpr int kRoundBatchMax = 8;

// Scratch of the fused round kernel, per round of a batch.
struct RoundScratch {
  double *partials;            // [round][2 n][blocks]
  double *group_partials;      // [round][2 n][groups]
  unsigned int *tickets;       // [1 + groups]: the launch's ticket, then one per group of blocks
  float *out_rounds;           // [round][2 kMaxDevices]: the statistics of every round of the batch
  float *out;                  // [2 kMaxDevices]: the statistics of the batch's last round
  // value `at` of round r of n_rounds
  __device__ __forceinline__ void put(int r, int n_rounds, int at, float x) const {
    float *out_r = out_rounds + r * 2 * kMaxDevices;
    if (access_ok(out_r + at, 4)) out_r[at] = x;
    if (r + 1 == n_rounds && access_ok(out + at, 4)) out[at] = x;
  }
};

template <typename WT, typename MT, typename Gen, int E, int RM, bool PF, int NR>
__global__ void __launch_bounds__(kThreads, PF ? kRoundBlocksPerSM - 1 : kRoundBlocksPerSM)
k_round(WT *__restrict__ w, MT *__restrict__ m, int64_t n_params, RoundBatch<NR> b, PhiloxKeys keys,
        StepConsts k, RoundScratch scratch) {
  constexpr bool kVote = !(sizeof(WT) == 2 && sizeof(MT) == 4 && RM == 0 && PF && NR > 1);  // (measured at step_noise)
  constexpr int kWarps = kThreads / 32;
  extern __shared__ float s_acc[];  // [n][kThreads]: per-thread row sums of the round in hand
  __shared__ double s_part[NR][2 * kMaxDevices];  // the block's sums, per round
  __shared__ bool s_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n_dev = b.round[0].n;
  for (int j = 0; j < n_dev; ++j) s_acc[j * kThreads + threadIdx.x] = 0.f;
  for (int t = threadIdx.x; t < NR * 2 * kMaxDevices; t += kThreads) (&s_part[0][0])[t] = 0.0;
  __syncthreads();

  const int64_t n_packs = (n_params + E - 1) / E;
  const int64_t n_chunks = (n_packs + kThreads - 1) / kThreads;
  for (int64_t chunk = blockIdx.x; chunk < n_chunks; chunk += gridDim.x) {
    // The chunk's work is compiled twice: for chunks whose packs are all full (`live` is then the
    // constant E, every ragged-tail test in the loads and stores folds away and stores are of 32 bytes)
    // and for the chunk that holds the end of the vector (and, there, the lanes beyond it), or all
    // chunks of an arena whose rows do not start at multiples of 32 bytes.
    auto do_chunk = [&](auto all_full) {
      const int64_t p = chunk * kThreads + threadIdx.x;
      const auto live = live_of<E>(all_full, n_params, p);
      const GroupProducts<E / 4> gp(p);
      char *wp = reinterpret_cast<char *>(w) + p * (int64_t)(E * sizeof(WT));
      char *mp = reinterpret_cast<char *>(m) + p * (int64_t)(E * sizeof(MT));

      auto do_round = [&](const RoundArgs &a, const int r) {
        // Row j as it is after its local steps: loads w (and m when the row runs steps), runs the
        // steps, stores the momentum, and leaves in wv what the row now holds (as stored; dead lanes
        // 0).  fp32 values are updated in the registers they were loaded into.
        // PF: the next row's loads are issued before this row's steps (see the kernel's header).
        RawPack<WT, E> rw_next;
        RawPack<MT, E> rm_next;
        auto fetch = [&](int j) {
          ld_raw(at_row<WT>(wp, a.r[j].w_off), live, rw_next);
          if (a.r[j].steps > 0) ld_raw(at_row<MT>(mp, a.r[j].m_off), live, rm_next);
        };
        if constexpr (PF) fetch(0);
        auto row_after_steps = [&](int j, float (&wv)[E]) -> bool {
          RawPack<WT, E> rw;
          RawPack<MT, E> rm;
          if constexpr (PF) {
            rw = rw_next;
            rm = rm_next;
            if (j + 1 < a.n) fetch(j + 1);
          } else {
            ld_raw(at_row<WT>(wp, a.r[j].w_off), live, rw);
          }
          const bool stepped = a.r[j].steps > 0;
          if (stepped) {
            if constexpr (!PF) ld_raw(at_row<MT>(mp, a.r[j].m_off), live, rm);
            float mv[E];
            unpack(rw, wv);
            unpack(rm, mv);
            sgd_steps<Gen, E / 4, kVote>(wv, mv, gp, a.r[j], keys, k);
            if constexpr (RM == 1) round_stochastic<MT, false>(wv, mv, gp, a.r[j], keys);
            st_pack_any(at_row<MT>(mp, a.r[j].m_off), 0, live, mv);
            if constexpr (RM == 0) {
#pragma unroll
              for (int i = 0; i < E; ++i) wv[i] = as_stored(wv[i], w);
            }
            if (live < E) {  // the ragged last pack of a row and the lanes beyond it: dead lanes stay 0
#pragma unroll
              for (int i = 0; i < E; ++i) wv[i] = i < live ? wv[i] : 0.f;
            }
          } else {
            unpack(rw, wv);
          }
          return stepped;
        };

        // ---- the selected devices in draw order: acc = a_0 w_0, then acc = fma(a_j, w_j, acc)
        float acc[E];
        {
          float wv[E];
          row_after_steps(0, wv);
          const float a0 = a.a[0];
#pragma unroll
          for (int i = 0; i < E; ++i) acc[i] = __fmul_rn(a0, wv[i]);
        }
        for (int j = 1; j < a.k; ++j) {
          float wv[E];
          row_after_steps(j, wv);
          const float aj = a.a[j];
#pragma unroll
          for (int i = 0; i < E; ++i) acc[i] = fmaf(aj, wv[i], acc[i]);
        }
        {
          float n2 = 0.f;
#pragma unroll
          for (int i = 0; i < E; ++i) {
            acc[i] = as_stored(acc[i], w);
            n2 = fmaf(acc[i], acc[i], n2);
          }
          // a single selected device that ran no steps already holds the aggregate (a_0 = 1)
          if (a.k > 1 || a.r[0].steps > 0)
            for (int t = 0; t < a.k; ++t) st_pack_any(at_row<WT>(wp, a.r[t].w_off), 0, live, acc);
          add_row_sums(s_acc, a.k - 1, n2, 0.f, lane);  // one value for all selected devices
        }
        // ---- the other devices: keep their own model, or receive the aggregate
        for (int j = a.k; j < a.n; ++j) {
          float wv[E];
          const bool stepped = row_after_steps(j, wv);
          if (a.write_all == 1) {
#pragma unroll
            for (int i = 0; i < E; ++i) wv[i] = acc[i];
          } else if (a.write_all == 2) {
#pragma unroll
            for (int i = 0; i < E; ++i)
              wv[i] = as_stored(fmaf(a.beta, acc[i], __fmul_rn(a.one_minus_beta, wv[i])), w);
          }
          if (stepped || a.write_all) st_pack_any(at_row<WT>(wp, a.r[j].w_off), 0, live, wv);
          float n2 = 0.f, d2 = 0.f;
#pragma unroll
          for (int i = 0; i < E; ++i) {
            const float d = wv[i] - acc[i];
            n2 = fmaf(wv[i], wv[i], n2);
            d2 = fmaf(d, d, d2);
          }
          add_row_sums(s_acc, j, n2, d2, lane);
        }
        // ---- block: fold the per-thread slots of every visit index j >= k - 1 into the block's
        // sums of this round and clear them.  Warp w takes the visit indices k - 1 + w,
        // k - 1 + w + 8, ...: each lane adds the slots of the threads that share its lane index
        // (one per warp, in warp order; lower half-warps hold norms, upper halves distances), then a
        // butterfly over the half-warp finishes the two sums.
        __syncthreads();
        for (int j = a.k - 1 + warp; j < a.n; j += kWarps) {
          double d = 0.0;
#pragma unroll
          for (int wi = 0; wi < kWarps; ++wi) {
            d += (double)s_acc[j * kThreads + wi * 32 + lane];
            s_acc[j * kThreads + wi * 32 + lane] = 0.f;
          }
#pragma unroll
          for (int off = 8; off > 0; off >>= 1) d += __shfl_xor_sync(0xFFFFFFFFu, d, off);
          if ((lane & 15) == 0) s_part[r][2 * j + (lane >> 4)] += d;  // value = 2 * visit index + which
        }
        __syncthreads();
      };
      // A launch of a single round reads its arguments at constant addresses (the compiler then
      // keeps the row descriptors on the uniform datapath); a batch indexes them by the round.
      if constexpr (NR == 1) {
        do_round(b.round[0], 0);
      } else {
        for (int r = 0; r < b.n_rounds; ++r) do_round(b.round[r], r);
      }
    };
    if ((chunk + 1) * kThreads * E <= n_params && rows_at_32(w, m))
      do_chunk(std::true_type{});
    else
      do_chunk(std::false_type{});
  }
  // ---- launch: partials[round][value][block], then one last-ticket finish for all rounds (one
  // fence and one ticket per block)
  const int n_rounds = NR == 1 ? 1 : b.n_rounds;
  const int n_vals = n_rounds * 2 * n_dev;
  for (int t = threadIdx.x; t < n_vals; t += kThreads) {
    const int r = NR == 1 ? 0 : t / (2 * n_dev);
    double *slot = scratch.partials + (int64_t)t * gridDim.x + blockIdx.x;
    if (access_ok(slot, 8)) *slot = s_part[r][t - r * 2 * n_dev];
  }
  finish_by_groups(scratch.partials, scratch.group_partials, n_vals, scratch.tickets + 1, scratch.tickets, &s_last,
                   [&](int t, double sum) {
    const int r = NR == 1 ? 0 : t / (2 * n_dev), v = t - r * 2 * n_dev, j = v >> 1, which = v & 1;
    const RoundArgs &a = b.round[r];
    auto put = [&](int at, float x) { scratch.put(r, n_rounds, at, x); };
    if (j == a.k - 1) {  // the selected devices share one norm and are at distance 0
      for (int q = 0; q < a.k; ++q) put(which * n_dev + a.r[q].row, which ? 0.f : (float)sum);
    } else if (j >= a.k) {
      put(which * n_dev + a.r[j].row, (float)sum);
    }
  });
}

// ------------------------------------------------------------------------------------------
// Fused rounds of small vectors: a warp per row.  The rows of a tile of 32 * E columns are spread over
// the warps of a group instead of being walked by one thread, and stay in registers through all rounds
// of a batch.  Per round a warp runs its row's steps; the selected warps leave their rows in shared
// memory; one barrier of the group; every warp then forms the aggregate for itself (in draw order, as
// k_round does) and takes its statistics against it.  Two buffers in turn make one barrier per round
// enough: a warp that writes round r + 2 has passed the barrier of round r + 1, which no warp reaches
// before it has read round r.  Parameters and momentum come out bit-identical to k_round.
// What bounds a round here is latency: that of the slowest row (k_round: of all rows one after the
// other) plus the hand-over, and there are n times as many warps to fill the chip.
// On large vectors the waits at the barrier, where all warps of a group are in the same phase, cost more
// than registers save; there k_round is the faster one (the host decides: see rows_form).
// A row moves to another warp from block to block, so that the heavy rows meet all SM sub-partitions.
// Sums of a row: the fp32 part of the order is k_round's (a thread's pack, then the lanes l and l ^ 16), fp64 beyond;
// the lanes' values wait in shared memory until the tile's rounds are done (a butterfly in each round stood between
// two barriers: 8 rounds of 4 devices and 100,000 parameters 3.77 -> 3.73 us each).
// ------------------------------------------------------------------------------------------
// Threads of a block, at most: the build for 512 has twice the registers, for batches whose blocks have an SM to
// themselves and for single rounds of the same vectors.
constexpr int kRowsMaxThreads = 1024, kRowsFewThreads = 512;

struct RowsStep {  // one device in one round
  int32_t steps;
  uint32_t base_lo, r1_c2;  // as in RowStep
  int32_t visit;            // position in the draw (0 .. k - 1: selected), or k and above
};
struct RowsUnits {  // the order of the tiles' sums
  int32_t tiles;             // are added first, to a unit's
  int32_t parts;             // units of a block of a batch
  int32_t per_block;         // units of a block of a single round
  int32_t n_units, n_sums;   // units of the vector, and blocks of a batch
};
template <int NR>
struct RowsBatch {
  int32_t n, k, n_rounds;
  int32_t groups;             // tiles that a block has in hand at a time
  RowsUnits units;            // (blocks of up to kRowsFewThreads)
  float beta, one_minus_beta;
  int32_t write_all[NR];      // as in RoundArgs
  float a[NR][kMaxDevices];   // aggregation weights in draw order
  __align__(16) RowsStep s[NR][kMaxDevices];
};

// A selected row of a tile in shared memory: [plane of 16 (or 8) bytes][lane].
template <typename WT, int E>
struct SelectedRow {
  static constexpr int kPackBytes = E * (int)sizeof(WT);
  using Unit = typename std::conditional<kPackBytes >= 16, uint4, uint2>::type;
  static constexpr int kPlanes = kPackBytes / (int)sizeof(Unit);
  static constexpr int kBytes = kPackBytes * 32;
  static __device__ __forceinline__ void load(const char *row, int lane, RawPack<WT, E> &r) {
    Unit u[kPlanes];
#pragma unroll
    for (int i = 0; i < kPlanes; ++i) u[i] = reinterpret_cast<const Unit *>(row)[i * 32 + lane];
    memcpy(&r, u, kPackBytes);
  }
  static __device__ __forceinline__ void store(char *row, int lane, const RawPack<WT, E> &r) {
    Unit u[kPlanes];
    memcpy(u, &r, kPackBytes);
#pragma unroll
    for (int i = 0; i < kPlanes; ++i) reinterpret_cast<Unit *>(row)[i * 32 + lane] = u[i];
  }
};

// Dynamic shared memory of a block: [group][2][k] selected rows, [group][round][n][2] row sums, [warp][round][32]
// what a row's lanes have to add in a tile.
__host__ __device__ constexpr int rows_slots(int rounds) { return (rounds + 3) / 4 * 4; }  // four rounds are added at a time
template <typename WT, int E>
constexpr size_t rows_selected_bytes(int k) { return (size_t)2 * k * SelectedRow<WT, E>::kBytes; }
template <typename WT, int E>
constexpr size_t rows_shared_bytes(int groups, int n, int k, int rounds) {
  return groups * (rows_selected_bytes<WT, E>(k) + sizeof(double) * 2 * n * rounds + sizeof(float) * 32 * n * rows_slots(rounds));
}

template <typename WT, typename MT, typename Gen, int E, int RM, int NR, int kMaxThreads>
__global__ void __launch_bounds__(kMaxThreads)
k_round_rows(WT *__restrict__ w, MT *__restrict__ m, int64_t stride, int64_t n_params,
             PhiloxKeys keys, StepConsts k, RoundScratch scratch, const __grid_constant__ RowsBatch<NR> b) {
  using Sel = SelectedRow<WT, E>;
  extern __shared__ __align__(16) char s_rows[];
  __shared__ bool s_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = b.n, n_sel = b.k, groups = b.groups;
  const int n_rounds = NR == 1 ? 1 : b.n_rounds;
  const int n_vals = n_rounds * 2 * n;
  const int group = warp / n;
  const int row = (warp - group * n + (int)blockIdx.x) % n;
  char *sel = s_rows + group * 2 * n_sel * Sel::kBytes;
  double *all_sums = reinterpret_cast<double *>(s_rows + groups * 2 * n_sel * Sel::kBytes);
  double *sums = all_sums + group * n_vals + 2 * row;  // each owned by the warp of that row
  float *slots = reinterpret_cast<float *>(all_sums + groups * n_vals) + warp * rows_slots(n_rounds) * 32;
  for (int t = threadIdx.x; t < groups * n_vals; t += blockDim.x) all_sums[t] = 0.0;
  RowStep rs;
  rs.row = row;
  {
    const uint64_t dp = (uint64_t)kPhiloxM1 * (uint32_t)row;
    rs.r1_c0 = (uint32_t)(dp >> 32) ^ keys.a[0];
    rs.r1_c1 = (uint32_t)dp;
  }
  __syncthreads();

  const int64_t n_packs = (n_params + E - 1) / E;
  const int64_t n_tiles = (n_packs + 31) / 32;
  // (warps beyond the groups' are there for the finish)
  for (int64_t tile = group < groups ? (int64_t)blockIdx.x * groups + group : n_tiles; tile < n_tiles;
       tile += (int64_t)gridDim.x * groups) {
    auto do_tile = [&](auto all_full) {
      const int64_t p = tile * 32 + lane;
      const auto live = live_of<E>(all_full, n_params, p);
      const GroupProducts<E / 4> gp(p);
      WT *wp = w + row * stride + p * E;
      MT *mp = m + row * stride + p * E;
      float wv[E], mv[E];
      {
        RawPack<WT, E> rw;
        RawPack<MT, E> rm;
        ld_raw(wp, live, rw);
        ld_raw(mp, live, rm);
        unpack(rw, wv);
        unpack(rm, mv);
      }
      bool w_changed = false, m_changed = false;
#pragma unroll 1
      for (int r = 0; r < n_rounds; ++r) {
        const RowsStep &st = b.s[r][row];
        rs.steps = st.steps;
        rs.base_lo = st.base_lo;
        rs.r1_c2 = st.r1_c2;
        const int j = st.visit, write_all = b.write_all[r];
        if (rs.steps > 0) {
          sgd_steps<Gen, E / 4>(wv, mv, gp, rs, keys, k);
          if constexpr (RM == 1) {
            round_stochastic<MT, false>(wv, mv, gp, rs, keys);
          } else {
#pragma unroll
            for (int i = 0; i < E; ++i) {
              wv[i] = as_stored(wv[i], w);
              mv[i] = as_stored(mv[i], m);
            }
          }
          if (live < E) {  // lanes beyond the end of the vector stay 0 in the sums
#pragma unroll
            for (int i = 0; i < E; ++i) wv[i] = i < live ? wv[i] : 0.f;
          }
          w_changed = m_changed = true;
        }
        char *buf = sel + (r & 1) * n_sel * Sel::kBytes;
        if (j < n_sel) {
          RawPack<WT, E> rw;
          pack_raw(wv, rw);
          Sel::store(buf + j * Sel::kBytes, lane, rw);
        }
        asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "r"(n * 32) : "memory");
        float acc[E];
        {
          RawPack<WT, E> rw;
          float v[E];
          Sel::load(buf, lane, rw);
          unpack(rw, v);
          const float a0 = b.a[r][0];
#pragma unroll
          for (int i = 0; i < E; ++i) acc[i] = __fmul_rn(a0, v[i]);
          for (int t = 1; t < n_sel; ++t) {
            Sel::load(buf + t * Sel::kBytes, lane, rw);
            unpack(rw, v);
            const float a_t = b.a[r][t];
#pragma unroll
            for (int i = 0; i < E; ++i) acc[i] = fmaf(a_t, v[i], acc[i]);
          }
        }
#pragma unroll
        for (int i = 0; i < E; ++i) acc[i] = as_stored(acc[i], w);
        if (j < n_sel ? n_sel > 1 || rs.steps > 0 : write_all == 1) {  // (see k_round for the single device without steps)
#pragma unroll
          for (int i = 0; i < E; ++i) wv[i] = acc[i];
          w_changed = true;
        } else if (j >= n_sel && write_all == 2) {
#pragma unroll
          for (int i = 0; i < E; ++i)
            wv[i] = as_stored(fmaf(b.beta, acc[i], __fmul_rn(b.one_minus_beta, wv[i])), w);
          w_changed = true;
        }
        float n2 = 0.f, d2 = 0.f;
#pragma unroll
        for (int i = 0; i < E; ++i) {
          const float d = wv[i] - acc[i];
          n2 = fmaf(wv[i], wv[i], n2);
          d2 = fmaf(d, d, d2);
        }
        const bool upper = (lane & 16) != 0;
        slots[r * 32 + lane] = (upper ? d2 : n2) + __shfl_xor_sync(0xFFFFFFFFu, upper ? n2 : d2, 16);
      }
      __syncwarp();
#pragma unroll 1
      for (int r0 = 0; r0 < n_rounds; r0 += 4) {  // 8 lanes per round: 4 add its norms, 4 its distances
        const float4 v = reinterpret_cast<const float4 *>(slots + r0 * 32)[lane];
        double d = ((double)v.x + (double)v.y) + ((double)v.z + (double)v.w);
        d += __shfl_xor_sync(0xFFFFFFFFu, d, 1);
        d += __shfl_xor_sync(0xFFFFFFFFu, d, 2);
        const int r = r0 + (lane >> 3);
        if ((lane & 3) == 0 && r < n_rounds) sums[r * 2 * n + ((lane >> 2) & 1)] += d;
      }
      if (w_changed) st_pack_any(wp, 0, live, wv);
      if (m_changed) st_pack_any(mp, 0, live, mv);
      // the next tile's first round must not overwrite a buffer that is still being read
      asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "r"(n * 32) : "memory");
    };
    if ((tile + 1) * 32 * E <= n_params && rows_at_32(w, m))
      do_tile(std::true_type{});
    else
      do_tile(std::false_type{});
  }
  __syncthreads();
  auto put = [&](int t, double sum) {
    const int r = t / (2 * n), v = t - r * 2 * n, at = (v & 1) * n + (v >> 1);  // [norms of the rows][distances]
    const bool holder = b.s[r][v >> 1].visit < n_sel;  // of the aggregate: at distance 0, whatever its values
    scratch.put(r, n_rounds, at, holder && (v & 1) ? 0.f : (float)sum);
  };
  if constexpr (kMaxThreads == kRowsFewThreads && NR == 1) {
    // the sums of a batch's blocks, which are not this launch's (see rows_units): the warps of a tile's rows store them
    const auto &u = b.units;
    const int at_unit = (int)blockIdx.x * u.per_block + group;
    if (group < u.per_block && at_unit < u.n_units && lane < 2) {
      const int t = 2 * (warp - group * n) + lane;
      const int sum = u.parts == 1 ? at_unit : u.parts == 2 ? at_unit / 2 : at_unit / 3;
      double d = 0.0;
      for (int g = group * u.tiles; g < (group + 1) * u.tiles; ++g) d += all_sums[g * n_vals + t];
      double *at = scratch.partials + (t * u.parts + at_unit - sum * u.parts) * u.n_sums + sum;
      if (access_ok(at, 8)) *at = d;
    }
    if (!is_last_block(scratch.tickets, gridDim.x, &s_last)) return;
    if (u.parts == 1)
      sum_up_to_four_groups(scratch.partials, n_vals, u.n_sums, put);
    else if (u.parts == 2)
      sum_parts<2>(scratch.partials, n_vals, u.n_units, u.n_sums, put);
    else
      sum_parts<3>(scratch.partials, n_vals, u.n_units, u.n_sums, put);
    if (threadIdx.x == 0) scratch.tickets[0] = 0u;
  } else {
    for (int t = threadIdx.x; t < n_vals; t += blockDim.x) {
      double d = 0.0;
      if (kMaxThreads == kRowsFewThreads) {
        for (int g0 = 0; g0 < groups; g0 += b.units.tiles) {
          double of_unit = 0.0;
          for (int g = g0; g < g0 + b.units.tiles; ++g) of_unit += all_sums[g * n_vals + t];
          d += of_unit;
        }
      } else {
        for (int g = 0; g < groups; ++g) d += all_sums[g * n_vals + t];
      }
      double *at = scratch.partials + (int64_t)t * gridDim.x + blockIdx.x;
      if (access_ok(at, 8)) *at = d;
    }
    // one finish over all rounds of the batch (one fence and one ticket per block)
    finish_by_groups(scratch.partials, scratch.group_partials, n_vals, scratch.tickets + 1, scratch.tickets, &s_last, put);
  }
}

// ------------------------------------------------------------------------------------------
// Several rounds per launch with the replicas on the SM ("resident" batch).  A block of 128 threads takes
// its columns through all rounds of the batch.  The rows are read from HBM once, live on the SM in between
// and are written back once: parameters in shared memory, momentum in tensor memory - 256 KB per SM
// that no kernel here needs for a contraction and that doubles what an SM can hold.  Rows that find no
// room stay in the arena, i.e. in L2.  Either way a value is only ever touched by the thread that owns its
// column, so no barrier separates the rows or rounds of a block.
// The arithmetic of a round is that of k_round, in the same order: same results bit for bit.
//
// What bounds it: on large vectors the row walk through L2 ran into the board's power cap (1000 W, SM clock
// down to 1600 - 1750 MHz); here a round moves a fraction of the bytes, keeps the full clock at 500 - 900 W
// and is bound by instruction latency at 3 to 6 warps per scheduler (237 instructions per row and pack at one step).
// How many blocks share an SM decides between warps to hide latency with and rows that find room (the
// host chooses).  Sustained, us per round of a batch of 8, row walk -> resident: 16 devices, 2^24, one
// step 496 -> 409 (before the 32-byte stores 3, 4, 5, 6 blocks: 424, 436, 431, 478), two steps at 14.7 M 635 -> 534 (574, 556, 534,
// 525); 8 devices, 11.2 M, one step 148 -> 124; 32 devices, 23.5 M 1955 -> 1574 (2, 3 blocks: 1830, 1599);
// bf16 parameters, 16 devices, 2^22 125 -> 108; 16 devices, 14.7 M, steps 1,1,2,2,4,4,8,8: 863 (one launch
// per round) -> 822 (3 .. 6 blocks: 935, 887, 844, 821).
// A round that overwrites all devices stores the aggregate and reads nothing: all rows share its norm (16
// devices, 12.8 M, steps 1,1,2,2,4,4,8,8, every round synchronised: 781 us per round with a read of every row
// before its store, 677 without; one launch per round 748).
// The first step's noise is drawn while the row's values are on their way (434 -> 421 us with everything on
// the SM, 16 devices).  Each row is either wholly on the SM or wholly in the arena and the code is compiled
// for either place: choosing at every access cost 100 instructions per row and pack in register copies.
// Values move between the arena and the SM as they are: NaNs of rows that nothing changes keep their bits.
// ------------------------------------------------------------------------------------------
constexpr int kResidentThreads = 128;
constexpr int kResidentMaxBlocks = 6;  // per SM: what the registers are bounded for (80 a thread; builds that use no more
                                       // than 72 could have 7); shared memory sets the actual number
constexpr int kResidentOneVisitMaxBlocks = 5;  // ... of the build with one visit per row and round, as far as rows make
                                               // room for each other: a sixth runs where there is room for as many rows

struct ResidentBatch {
  int32_t n, k, n_rounds;
  int32_t n_on_chip;  // devices 0 .. n_on_chip - 1 live on the SM, the others in the arena
  float beta, one_minus_beta;
  int32_t write_all[kRoundBatchMax];                // as in RoundArgs
  int32_t first_store[kRoundBatchMax];              // 1 where a single selected device holds the aggregate already
  int32_t n_stepping[kRoundBatchMax];               // devices that run at least one step ...
  int32_t order[kRoundBatchMax][kMaxDevices];       // ... by descending step count
  int32_t draw[kRoundBatchMax][kMaxDevices];        // devices: the selected ones in draw order, then the rest
  float a[kRoundBatchMax][kMaxDevices];             // aggregation weights in draw order
  uint32_t r1_c0[kMaxDevices], r1_c1[kMaxDevices];  // as in RowStep
  int64_t w_off[kMaxDevices], m_off[kMaxDevices];   // as in RowStep
  RowsStep s[kRoundBatchMax][kMaxDevices];          // (visit is not used)
};

// A thread's packs in shared memory: [row][plane of 16 bytes][thread].
template <typename WT>
struct RowStore {
  static constexpr int kPackBytes = 8 * (int)sizeof(WT);
  static constexpr int kPlanes = kPackBytes / 16;
  static constexpr int kRowBytes = kPackBytes * kResidentThreads;
  static __device__ __forceinline__ void load(const char *mine, int row, RawPack<WT, 8> &r) {
    uint4 u[kPlanes];
#pragma unroll
    for (int i = 0; i < kPlanes; ++i)
      u[i] = *reinterpret_cast<const uint4 *>(mine + row * kRowBytes + i * 16 * kResidentThreads);
    memcpy(&r, u, kPackBytes);
  }
  static __device__ __forceinline__ void store(char *mine, int row, const RawPack<WT, 8> &r) {
    uint4 u[kPlanes];
    memcpy(u, &r, kPackBytes);
#pragma unroll
    for (int i = 0; i < kPlanes; ++i)
      *reinterpret_cast<uint4 *>(mine + row * kRowBytes + i * 16 * kResidentThreads) = u[i];
  }
};

// Tensor memory as per-thread storage: a warp owns the 32 lanes of its quarter, a thread one lane; a pack
// is 4 or 8 consecutive 32-bit columns of that lane.  A load is complete after tmem_wait_load (the values
// pass through tmem_use there, so that nothing reads them before), a store is visible to the thread's
// later loads after tmem_wait_store.
__device__ __forceinline__ void tmem_load(uint32_t at, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(at));
}
__device__ __forceinline__ void tmem_load(uint32_t at, uint32_t (&v)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(at));
}
__device__ __forceinline__ void tmem_store(uint32_t at, const uint32_t (&v)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(at), "r"(v[0]), "r"(v[1]),
               "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}
__device__ __forceinline__ void tmem_store(uint32_t at, const uint32_t (&v)[4]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(at), "r"(v[0]), "r"(v[1]), "r"(v[2]),
               "r"(v[3]) : "memory");
}
__device__ __forceinline__ void tmem_wait_load() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_store() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void tmem_use(uint32_t (&v)[N]) {
#pragma unroll
  for (int i = 0; i < N; ++i) asm volatile("" : "+r"(v[i]));
}

// Columns of tensor memory that hold n packs of `words` words: a power of two, 32 at least.
__host__ __device__ constexpr int tmem_columns(int n, int words) {
  int c = 32;
  while (c < n * words) c *= 2;
  return c;
}

// Row sums of a warp that no other warp takes part in: the fp32 part of the order is k_round's (a
// thread's pack, then the lanes l and l ^ 16), the rest is added in fp64, as there.  add() leaves 32 values
// per row in the warp's slots, fold() adds those of up to 4 rows: 8 lanes per row.
struct WarpRowSums {
  static constexpr int kRows = 4;
  static constexpr int kFloats = kRows * 32;
  static __device__ __forceinline__ void add(float *slots, int s, float n2, float d2, int lane) {
    const bool upper = (lane & 16) != 0;
    const float keep = upper ? d2 : n2, give = upper ? n2 : d2;
    slots[s * 32 + lane] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, 16);
  }
  // sums of the visit indices j0 .. j0 + count - 1 -> line[2 j + which]
  static __device__ __forceinline__ void fold(const float *slots, int j0, int count, double *line, int lane) {
    __syncwarp();
    const float4 v = reinterpret_cast<const float4 *>(slots)[lane];
    double d = ((double)v.x + (double)v.y) + ((double)v.z + (double)v.w);
    d += __shfl_xor_sync(0xFFFFFFFFu, d, 1);
    d += __shfl_xor_sync(0xFFFFFFFFu, d, 2);
    if ((lane & 3) == 0 && (lane >> 3) < count) line[2 * j0 + (lane >> 2)] = d;
    __syncwarp();
  }
};

// Shared memory of a block beside its rows: [warp][round][2 n] sums and the warps' slots.
constexpr size_t resident_sums_bytes(int n, int rounds) {
  return (kResidentThreads / 32) * (sizeof(double) * 2 * n * rounds + sizeof(float) * WarpRowSums::kFloats);
}

// The builds of the kernel: all rows on the SM; a part of them; a part of them, and one visit per row and round.
// With visits apart - steps of all rows, aggregation, sums - a row that lives in L2 crosses to the SM and back up to
// three times a round; with one, in draw order, once, and a selected row is stored only as the aggregate, but the
// aggregate and the row's sums then take registers through the steps: with several steps per row, where warps to
// hide latency with count for more, or with all rows on the SM, that costs more than it saves.  Sustained, us per
// round of a batch of 8, apart / one visit: 16 devices, 2^24, one step 406 / 387, 2^22 112.4 / 107.3; 32 devices,
// 2^22 300 / 282; 16 devices, 2^24, two steps 590 / 587; 14.7 M, steps 1,1,2,2,4,4,8,8 809 / 831; all rows on the SM, 8
// devices, 11.2 M, one step 118 / 121; bf16 parameters, 16 devices, 2^22, one step 102 / 107.  Fewer rows on the SM for a
// sixth block lose (2^24, one step 397), but where short batches' sums leave room for one with the same rows it gains; with 5
// / 6: 16 devices, 2^24, 2 rounds, one step 511 / 490, 14 devices, 3 rounds 385 / 355, 9 devices, 4 rounds 236 / 218.
enum class Resident { kAll, kPart, kPartOneVisit };
constexpr int resident_max_blocks(Resident form) {
  return form == Resident::kPartOneVisit ? kResidentOneVisitMaxBlocks : kResidentMaxBlocks;
}

template <typename WT, typename MT, typename Gen, int RM, Resident kForm>
__global__ void __launch_bounds__(kResidentThreads, resident_max_blocks(kForm))
k_rounds_resident(WT *__restrict__ w, MT *__restrict__ m, int64_t n_params, PhiloxKeys keys,
                  StepConsts k, RoundScratch scratch, const __grid_constant__ ResidentBatch b) {
  constexpr int E = 8, kWarps = kResidentThreads / 32;
  constexpr bool kAllOnChip = kForm == Resident::kAll;
  constexpr int kWords = E * (int)sizeof(MT) / 4;  // tensor memory columns per row
  using Store = RowStore<WT>;
  using Sums = WarpRowSums;
  extern __shared__ __align__(16) char s_raw[];
  __shared__ uint32_t s_tmem;
  __shared__ bool s_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = b.n, n_sel = b.k, n_on_chip = kAllOnChip ? n : b.n_on_chip;
  const int n_vals = b.n_rounds * 2 * n;
  char *mine = s_raw + 16 * threadIdx.x;                                        // [row][plane][thread]
  double *lines = reinterpret_cast<double *>(s_raw + n_on_chip * Store::kRowBytes);  // [warp][round][2 n]
  float *slots = reinterpret_cast<float *>(lines + kWarps * n_vals) + warp * Sums::kFloats;

  const int cols = tmem_columns(n_on_chip, kWords);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(&s_tmem)), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tm = s_tmem + ((uint32_t)warp << 21);  // this warp's quarter: lanes 32 * warp ...

  const int64_t n_packs = (n_params + E - 1) / E;
  const int64_t n_chunks = (n_packs + kResidentThreads - 1) / kResidentThreads;
  for (int64_t chunk = blockIdx.x; chunk < n_chunks; chunk += gridDim.x) {
    auto do_chunk = [&](auto all_full) {
      const int64_t p = chunk * kResidentThreads + threadIdx.x;
      const auto live = live_of<E>(all_full, n_params, p);
      const GroupProducts<E / 4> gp(p);
      char *wp = reinterpret_cast<char *>(w) + p * (int64_t)(E * sizeof(WT));
      char *mp = reinterpret_cast<char *>(m) + p * (int64_t)(E * sizeof(MT));
      // The lanes of a warp together, which the instructions on tensor memory want: what a chunk with the end of the
      // vector does under its lanes' conditions may leave them apart.
      auto together = [&]() {
        if constexpr (!decltype(all_full)::value) __syncwarp();
      };
      // A row's packs where they live; `where` is std::true_type for the SM, std::false_type for the arena.
      auto load_w = [&](auto where, int row, RawPack<WT, E> &r) {
        if constexpr (decltype(where)::value)
          Store::load(mine, row, r);
        else
          ld_raw(at_row<WT>(wp, b.w_off[row]), live, r);
      };
      auto store_w = [&](auto where, int row, const RawPack<WT, E> &r) {
        if constexpr (decltype(where)::value)
          Store::store(mine, row, r);
        else
          st_raw(at_row<WT>(wp, b.w_off[row]), live, r);
      };
      auto load_m = [&](auto where, int row, RawPack<MT, E> &r) {  // there after m_arrived
        if constexpr (decltype(where)::value) {
          uint32_t v[kWords];
          together();
          tmem_load(tm + row * kWords, v);
          memcpy(&r, v, sizeof(v));
        } else {
          ld_raw(at_row<MT>(mp, b.m_off[row]), live, r);
        }
      };
      auto m_arrived = [&](auto where, RawPack<MT, E> &r) {
        if constexpr (decltype(where)::value) {
          uint32_t v[kWords];
          together();
          tmem_wait_load();
          memcpy(v, &r, sizeof(v));
          tmem_use(v);
          memcpy(&r, v, sizeof(v));
        }
      };
      auto store_m = [&](auto where, int row, const RawPack<MT, E> &r) {
        if constexpr (decltype(where)::value) {
          uint32_t v[kWords];
          memcpy(v, &r, sizeof(v));
          together();
          tmem_store(tm + row * kWords, v);
        } else {
          st_raw(at_row<MT>(mp, b.m_off[row]), live, r);
        }
      };
      // A row's parameters as they stand, dead lanes 0.
      auto values = [&](auto where, int row, float (&wv)[E]) {
        RawPack<WT, E> r;
        load_w(where, row, r);
        unpack(r, wv);
        if (live < E) {
#pragma unroll
          for (int i = 0; i < E; ++i) wv[i] = i < live ? wv[i] : 0.f;
        }
      };
      // f for a row, compiled for either place (a choice at every access costs copies of the registers)
      auto at_place = [&](int row, auto f) {
        if (kAllOnChip || row < n_on_chip)
          f(std::true_type{}, row);
        else if constexpr (!kAllOnChip)
          f(std::false_type{}, row);
      };

      // ---- the rows come in
#pragma unroll 1
      for (int row = 0; row < n_on_chip; ++row) {
        RawPack<WT, E> rw;
        RawPack<MT, E> rm;
        ld_raw(at_row<WT>(wp, b.w_off[row]), live, rw);
        load_m(std::false_type{}, row, rm);
        store_w(std::true_type{}, row, rw);
        store_m(std::true_type{}, row, rm);
      }
      together();
      tmem_wait_store();

#pragma unroll 1
      for (int r = 0; r < b.n_rounds; ++r) {
        double *line = lines + (warp * b.n_rounds + r) * 2 * n;
        const int write_all = b.write_all[r];
        float acc[E];
        int slot = 0;
        // The steps of a row, from where it lives to registers; the momentum goes back at once.
        auto steps_of = [&](auto where, int row, float (&wv)[E]) {
          RowStep rs;
          rs.row = row;
          rs.steps = b.s[r][row].steps;
          rs.base_lo = b.s[r][row].base_lo;
          rs.r1_c2 = b.s[r][row].r1_c2;
          rs.r1_c0 = b.r1_c0[row];
          rs.r1_c1 = b.r1_c1[row];
          uint32_t c2_first[E / 4];
#pragma unroll
          for (int g = 0; g < E / 4; ++g) c2_first[g] = gp.hi[g] ^ rs.r1_c2;
          float mv[E];
          RawPack<WT, E> rw;
          RawPack<MT, E> rm;
          load_m(where, row, rm);
          load_w(where, row, rw);
          // the values are on their way while the first step's noise is drawn
          float2 nz[E / 4][2];
          step_noise<Gen, E / 4>(nz, 0, c2_first, gp, rs, keys, k);
          m_arrived(where, rm);
          unpack(rm, mv);
          unpack(rw, wv);
          step_update<E / 4>(wv, mv, nz, k);
#pragma unroll 1
          for (int e = 1; e < rs.steps; ++e) {
            step_noise<Gen, E / 4>(nz, e, c2_first, gp, rs, keys, k);
            step_update<E / 4>(wv, mv, nz, k);
          }
          if constexpr (RM == 1) round_stochastic<MT, true>(wv, mv, gp, rs, keys);
          pack_raw(mv, rm);
          store_m(where, row, rm);
        };
        // Aggregation in draw order: acc = a_0 w_0, then acc = fma(a_j, w_j, acc)
        auto start_aggregate = [&](const float (&wv)[E]) {
          const float a0 = b.a[r][0];
#pragma unroll
          for (int i = 0; i < E; ++i) acc[i] = __fmul_rn(a0, wv[i]);
        };
        auto add_selected = [&](int j, const float (&wv)[E]) {
          const float aj = b.a[r][j];
#pragma unroll
          for (int i = 0; i < E; ++i) acc[i] = fmaf(aj, wv[i], acc[i]);
        };
        // The aggregate goes to the first n_holders devices of the draw.
        auto hand_out = [&](int n_holders) {
          float n2 = 0.f;
#pragma unroll
          for (int i = 0; i < E; ++i) {
            acc[i] = as_stored(acc[i], w);
            n2 = fmaf(acc[i], acc[i], n2);
          }
          float d2_held = 0.f;  // of the devices that are overwritten: as (acc - acc)^2, NaN where acc is not finite
          if (write_all == 1) {
#pragma unroll
            for (int i = 0; i < E; ++i) d2_held = fmaf(acc[i], 0.f, d2_held);
          }
          RawPack<WT, E> ra;
          pack_raw(acc, ra);
#pragma unroll 1
          for (int t = b.first_store[r]; t < n_holders; ++t)
            at_place(b.draw[r][t], [&](auto where, int row) { store_w(where, row, ra); });
          Sums::add(slots, 0, n2, d2_held, lane);  // one value for all holders
        };
        auto mix = [&](float (&wv)[E]) {
#pragma unroll
          for (int i = 0; i < E; ++i)
            wv[i] = as_stored(fmaf(b.beta, acc[i], __fmul_rn(b.one_minus_beta, wv[i])), w);
        };
        auto add_sums = [&](int j, float s2, float d2) {
          if (++slot == Sums::kRows) {
            Sums::fold(slots, j - Sums::kRows, Sums::kRows, line, lane);
            slot = 0;
          }
          Sums::add(slots, slot, s2, d2, lane);
        };
        auto row_sums = [&](const float (&wv)[E], float &s2, float &d2) {
          s2 = d2 = 0.f;
#pragma unroll
          for (int i = 0; i < E; ++i) {
            const float d = wv[i] - acc[i];
            s2 = fmaf(wv[i], wv[i], s2);
            d2 = fmaf(d, d, d2);
          }
        };
        if constexpr (kForm == Resident::kPartOneVisit) {
#pragma unroll
          for (int i = 0; i < E; ++i) acc[i] = -0.f;  // fma(a, w, -0) is a w, whatever its sign
#pragma unroll 1
          for (int j = 0; j < n; ++j)
            at_place(b.draw[r][j], [&](auto where, int row) {
              float wv[E];
              const bool stepped = b.s[r][row].steps > 0;
              if (stepped) {
                steps_of(where, row, wv);
#pragma unroll
                for (int i = 0; i < E; ++i) wv[i] = as_stored(wv[i], w);
                if (live < E) {
#pragma unroll
                  for (int i = 0; i < E; ++i) wv[i] = i < live ? wv[i] : 0.f;
                }
              } else {
                values(where, row, wv);
              }
              if (j < n_sel) {
                add_selected(j, wv);
                if (j == n_sel - 1) hand_out(n_sel);
              } else {
                if (write_all == 2) mix(wv);
                if (write_all == 1) {
#pragma unroll
                  for (int i = 0; i < E; ++i) wv[i] = acc[i];
                }
                if (stepped || write_all) {
                  RawPack<WT, E> rw;
                  pack_raw(wv, rw);
                  store_w(where, row, rw);
                }
                if (write_all != 1) {
                  float s2, d2;
                  row_sums(wv, s2, d2);
                  add_sums(j, s2, d2);
                }
              }
            });
        } else {
          // ---- local steps
          const int n_step = b.n_stepping[r];
#pragma unroll 1
          for (int j = 0; j < n_step; ++j)
            at_place(b.order[r][j], [&](auto where, int row) {
              float wv[E];
              steps_of(where, row, wv);
              RawPack<WT, E> rw;
              pack_raw(wv, rw);
              store_w(where, row, rw);
            });
          // ---- aggregation with write-back
          at_place(b.draw[r][0], [&](auto where, int row) {
            float wv[E];
            values(where, row, wv);
            start_aggregate(wv);
          });
#pragma unroll 1
          for (int j = 1; j < n_sel; ++j)
            at_place(b.draw[r][j], [&](auto where, int row) {
              float wv[E];
              values(where, row, wv);
              add_selected(j, wv);
            });
          const int n_holders = write_all == 1 ? n : n_sel;
          hand_out(n_holders);
          // ---- the other devices: keep their own model, or mix the aggregate into it
#pragma unroll 1
          for (int j = n_holders; j < n; ++j) {
            float s2, d2;
            at_place(b.draw[r][j], [&](auto where, int row) {
              float wv[E];
              values(where, row, wv);
              if (write_all) {
                mix(wv);
                RawPack<WT, E> rw;
                pack_raw(wv, rw);
                store_w(where, row, rw);
              }
              row_sums(wv, s2, d2);
            });
            add_sums(j, s2, d2);
          }
        }
        Sums::fold(slots, write_all == 1 ? n_sel - 1 : n - 1 - slot, slot + 1, line, lane);
        together();
        tmem_wait_store();
      }

      // ---- the rows go back
#pragma unroll 1
      for (int row = 0; row < n_on_chip; ++row) {
        RawPack<WT, E> rw;
        RawPack<MT, E> rm;
        load_m(std::true_type{}, row, rm);
        load_w(std::true_type{}, row, rw);
        m_arrived(std::true_type{}, rm);
        st_raw(at_row<WT>(wp, b.w_off[row]), live, rw);
        store_m(std::false_type{}, row, rm);
      }
    };
    if ((chunk + 1) * kResidentThreads * E <= n_params && rows_at_32(w, m))
      do_chunk(std::true_type{});
    else
      do_chunk(std::false_type{});
    // devices that hold the aggregate share one sum
    auto has_sum = [&](int t) {
      const int r = t / (2 * n), j = (t - r * 2 * n) >> 1;
      return j >= n_sel - 1 && (j < n_sel || b.write_all[r] != 1);
    };
    __syncthreads();
    for (int t = threadIdx.x; t < n_vals; t += kResidentThreads) {  // a value belongs to one thread
      double *at = scratch.partials + (int64_t)t * gridDim.x + blockIdx.x;
      double sum = chunk == blockIdx.x || !access_ok(at, 8) ? 0.0 : *at;
      if (has_sum(t))
        for (int wi = 0; wi < kWarps; ++wi) sum += lines[wi * n_vals + t];
      if (access_ok(at, 8)) *at = sum;
    }
    __syncthreads();
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(cols));

  finish_by_groups(scratch.partials, scratch.group_partials, n_vals, scratch.tickets + 1, scratch.tickets, &s_last,
                   [&](int t, double sum) {
    const int r = t / (2 * n), v = t - r * 2 * n, j = v >> 1, which = v & 1;
    auto put = [&](int at, float x) { scratch.put(r, b.n_rounds, at, x); };
    if (j == n_sel - 1) {  // the holders of the aggregate share one norm; the selected ones are at distance 0
      for (int q = 0; q < (b.write_all[r] == 1 ? n : n_sel); ++q)
        put(which * n + b.draw[r][q], which && q < n_sel ? 0.f : (float)sum);
    } else if (j >= n_sel && b.write_all[r] != 1) {
      put(which * n + b.draw[r][j], (float)sum);
    }
  });
}

// ------------------------------------------------------------------------------------------
// Backup snapshot of a bf16 row, widened to fp32.  Bound by memory (6 bytes per parameter), and small beside
// the transfer that follows it.  dst is an allocation's start.
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads)
k_widen(const __nv_bfloat16 *__restrict__ src, float *__restrict__ dst, int64_t count) {
  const int64_t p = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  const int live = live_of(count, p, 8);
  if (live == 0) return;
  RawPack<__nv_bfloat16, 8> r;
  float v[8];
  ld_raw(src + 8 * p, live, r);
  unpack(r, v);
  if (live == 8)
    st_pack_any(dst, p, FullPack<8>{}, v);
  else
    st_pack_any(dst, p, live, v);
}

// ------------------------------------------------------------------------------------------
// Generator diagnostics.
// ------------------------------------------------------------------------------------------
__global__ void k_debug_philox(const uint32_t *__restrict__ ctr, PhiloxKeys keys, int64_t n,
                               uint32_t *__restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t c0 = ctr[4 * i], c1 = ctr[4 * i + 1], c2 = ctr[4 * i + 2], c3 = ctr[4 * i + 3];
  philox4x32_10(c0, c1, c2, c3, keys);
  out[4 * i] = c0; out[4 * i + 1] = c1; out[4 * i + 2] = c2; out[4 * i + 3] = c3;
}

template <typename Gen>
__global__ void k_debug_normals(const uint32_t *__restrict__ groups, int64_t n, uint32_t c1,
                                uint32_t c2, uint32_t c3, PhiloxKeys keys,
                                float4 *__restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  out[i] = normals_of_block<Gen>(groups[i], c1, c2, c3, keys);
}

}  // namespace hadfl
