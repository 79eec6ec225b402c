// Amax-history reduction and scale update as device functions: by a whole block in the standalone commit kernel and in the
// tail of a weight's cast (its last block), by one warp in the GEMM launches (X and G at a launch's start, where an earlier
// kernel has completed the amax; Y by the last CTA of the launch that computes it).  No launch is spent on a commit.
//   hist[c][count mod H] = amax;  scale_c = fp8_max / max(hist[c]) / 2^margin;  scale_inv_c = 1 / scale_c
// The block form: 256 threads, 64 per tensor class, all four classes in parallel, one barrier.  The ring's maximum is kept
// beside it so that a commit usually reads one entry instead of H.  The maximum is taken on
// the bit patterns of the non-negative FP32 entries, which orders them like their values and lets a NaN or Inf
// entry surface as "not finite" (scale then stays as it was, like for an all-zero window).
#pragma once
#include <cfloat>

#include "kernels.h"

namespace qe {

// Programmatic dependent launch.  Every kernel of the library is launched with programmatic stream serialization, so
// the next kernel in the stream may be scheduled while this one drains.  grid_dep_wait() returns once every kernel
// this one depends on has completed and its writes are visible: it must precede the first access to anything a
// predecessor produced.  grid_dep_launch() lets the successor's blocks start (they stop at their own wait).
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class Sync>
__device__ __forceinline__ void commit_classes(const CommitParams& p, int tid, uint32_t* red /* shared, 8 words */,
                                               Sync sync) {
  DevState* st = p.st;
  const int c = tid >> 6, g = tid & 63;
  const bool active = (p.class_mask >> c) & 1u;
  uint32_t m = 0, newest = 0, cnt = 0, pos = 0;
  uint32_t* h = reinterpret_cast<uint32_t*>(p.hist + (size_t)c * p.H);
  if (active) {
    cnt = __ldcg(&st->count[c]);
    newest = p.amax_override ? (__float_as_uint(__ldcg(p.amax_override)) & 0x7fffffffu) : __ldcg(&st->pending_amax[c]);
    const uint32_t wmax = __ldcg(&st->wmax[c]);  // maximum of the ring as it stands
    pos = cnt % p.H;
    const uint32_t evicted = __ldcg(h + pos);
    // The new maximum is known without reading the ring unless the entry that leaves was the maximum and the one
    // that enters is smaller: only then is the ring scanned (exactly the same value either way).
    if (newest >= wmax) m = newest;
    else if (evicted < wmax) m = wmax;
    else
      for (uint32_t i = g; i < p.H; i += 64) m = max(m, i == pos ? newest : __ldcg(h + i));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((tid & 31) == 0) red[tid >> 5] = m;
  sync();
  if (active && g == 0) {
    m = max(red[2 * c], red[2 * c + 1]);
    h[pos] = newest;
    st->count[c] = cnt + 1;
    st->pending_amax[c] = 0;
    st->wmax[c] = m;
    if (m != 0 && m < 0x7f800000u) {
      const float fp8_max = c == 2 ? 57344.0f : 448.0f;  // class 2 = gradients (E5M2), others E4M3
      float s = __fmul_rn(__fdiv_rn(fp8_max, __uint_as_float(m)), p.pow2_neg_margin);
      if (isinf(s)) s = FLT_MAX;
      st->scale[c] = s;
      st->scale_inv[c] = __fdiv_rn(1.0f, s);
    }
  }
  if (tid == 0 && p.bump_token) st->token += 1ull;
}

// The same commit done by ONE warp, class after class (a GEMM launch hands it one: X or G at its start, Y in its tail).
// A grouped launch may carry sixteen problems, each committed by a warp of its own, side by side: a commit is a chain of
// dependent global accesses, and one after the other the commits of a launch took as long as its tiles.  The rare ring
// scan takes 16-byte loads over all lanes, eight in flight each: F, dI and dW of a 256 x 256 x 256 linear plus the boundary
// take 57 us when no commit scans; when all three do, 62 us at 4096 entries (81 with 4-byte loads of eight lanes) and the
// same as without at 1024 (60).  Same values as commit_classes; the token is bumped atomically because two problems of
// one launch may belong to the same layer (its forward and its input gradient of different microbatches).
__device__ __forceinline__ uint32_t ring_max(const uint32_t* h, uint32_t H, uint32_t pos, uint32_t newest, uint32_t lane) {
  uint32_t m = newest, at = 0;  // (the entry at pos is the one that leaves)
  if ((reinterpret_cast<uintptr_t>(h) & 15u) == 0) {
    at = H & ~3u;
#pragma unroll 8
    for (uint32_t i = 4 * lane; i < at; i += 128) {
      const uint4 q = __ldcg(reinterpret_cast<const uint4*>(h + i));
      m = max(m, max(max(i == pos ? 0u : q.x, i + 1 == pos ? 0u : q.y), max(i + 2 == pos ? 0u : q.z, i + 3 == pos ? 0u : q.w)));
    }
  }
#pragma unroll 8
  for (uint32_t i = at + lane; i < H; i += 32) {
    const uint32_t q = __ldcg(h + i);
    m = max(m, i == pos ? 0u : q);
  }
  return __reduce_max_sync(0xffffffffu, m);
}

__device__ __forceinline__ void commit_classes_warp(const CommitParams& p, int lane) {
  DevState* st = p.st;
#pragma unroll 1
  for (uint32_t left = p.class_mask; left; left &= left - 1) {
    const int c = __ffs(left) - 1;
    uint32_t* h = reinterpret_cast<uint32_t*>(p.hist + (size_t)c * p.H);
    const uint32_t cnt = __ldcg(&st->count[c]);
    const uint32_t newest = p.amax_override ? (__float_as_uint(__ldcg(p.amax_override)) & 0x7fffffffu) : __ldcg(&st->pending_amax[c]);
    const uint32_t wmax = __ldcg(&st->wmax[c]);
    const uint32_t pos = cnt % p.H;
    const uint32_t evicted = __ldcg(h + pos);
    const uint32_t m = newest >= wmax ? newest : evicted < wmax ? wmax : ring_max(h, p.H, pos, newest, (uint32_t)lane);
    __syncwarp();  // every lane has read the entry that lane 0 replaces
    if (lane == 0) {
      h[pos] = newest;
      st->count[c] = cnt + 1;
      st->pending_amax[c] = 0;
      st->wmax[c] = m;
      if (m != 0 && m < 0x7f800000u) {
        const float fp8_max = c == 2 ? 57344.0f : 448.0f;
        float s = __fmul_rn(__fdiv_rn(fp8_max, __uint_as_float(m)), p.pow2_neg_margin);
        if (isinf(s)) s = FLT_MAX;
        st->scale[c] = s;
        st->scale_inv[c] = __fdiv_rn(1.0f, s);
      }
    }
  }
  if (lane == 0 && p.bump_token) atomicAdd(&st->token, 1ull);
}

// Returns true in every thread of exactly one block of the grid: the last one to get here.  Stores and atomics the
// grid made before this call are visible to that block afterwards.
template <class Sync>
__device__ __forceinline__ bool last_block(uint32_t* ticket, uint32_t nblocks, int tid, uint32_t* flag /* shared */,
                                           Sync sync) {
  __threadfence();
  sync();
  if (tid == 0) {
    const uint32_t t = atomicAdd(ticket, 1u);
    const bool last = t == nblocks - 1;
    if (last) atomicExch(ticket, 0u);  // ready for the next kernel that uses it
    *flag = last ? 1u : 0u;
  }
  sync();
  const bool last = *flag != 0u;
  if (last) __threadfence();
  return last;
}

}  // namespace qe
