// Amax-history reduction and scale update as device functions: by a whole block in the standalone commit kernel and in the
// tail of a weight's cast (its last block), by one warp or lane in the GEMM launches (X and G at a launch's start, where an earlier
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
// predecessor produced (or, for a cast that may overlap it, an acquire of its commits: Announce).  grid_dep_launch() lets the
// successor's blocks start (they stop at their own wait).
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

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

// Largest entry of a ring without the one at `hole`, by one warp: 16-byte loads over all lanes, four in flight each.
__device__ __forceinline__ uint32_t ring_max(const uint32_t* ring, uint32_t n, uint32_t hole, int lane) {
  uint32_t top = 0;
  auto take = [&](uint32_t i, uint32_t q) { top = max(top, i == hole ? 0u : q); };
  const uint32_t head = min(n, (4u - ((uint32_t)(reinterpret_cast<uintptr_t>(ring) >> 2) & 3u)) & 3u);  // up to a 16-byte boundary
  const uint32_t vecs = (n - head) / 4, tail = n - head - 4 * vecs;
  if ((uint32_t)lane < head) take((uint32_t)lane, __ldcg(ring + lane));
  if ((uint32_t)lane < tail) take(n - tail + (uint32_t)lane, __ldcg(ring + n - tail + lane));
#pragma unroll 4
  for (uint32_t v = (uint32_t)lane; v < vecs; v += 32) {
    const uint32_t i = head + 4 * v;
    const uint4 q = __ldcg(reinterpret_cast<const uint4*>(ring + i));
    take(i, q.x), take(i + 1, q.y), take(i + 2, q.z), take(i + 3, q.w);
  }
  return __reduce_max_sync(0xffffffffu, top);
}

// What a commit of a class reads besides its amax.
struct RingState {
  uint32_t count = 0, wmax = 0, evicted = 0;
};
__device__ __forceinline__ RingState ring_state(const CommitParams& p, int c) {
  RingState s;
  s.count = __ldcg(&p.st->count[c]);
  s.wmax = __ldcg(&p.st->wmax[c]);
  s.evicted = __ldcg(reinterpret_cast<const uint32_t*>(p.hist + (size_t)c * p.H) + s.count % p.H);
  return s;
}

// The same commit of ONE class (class_mask has one bit: X or G at a GEMM launch's start, Y in its tail) by one warp; EACH: of a
// class per lane, for lanes with `active`.  A grouped launch may carry dozens of problems, all committed side by side by lanes
// of the epilogue's warps: a commit is a chain of dependent global accesses, and one after the other the commits of a launch
// took as long as its tiles.  The code runs once per launch, from cold instruction memory, so it is short, with one loop for
// the rare ring scan, which a whole warp makes for one lane after the other (launches of one problem keep the form without
// lanes: with it twelve chained linears of 256 x 256 took 1402 us a step, without it 1389).  F, dI and dW of a 256 x 256 x 256
// linear plus the boundary take 55 us when no commit scans; when all three do, 60 us at 4096 entries and the same as without
// at 1024.  Same values as commit_classes; the token is bumped atomically because two problems of one launch may belong to
// the same layer (its forward and its input gradient of different microbatches).  `ahead`: the class's state, read after
// grid_dep_wait() and with no other commit of the class between that and this one.
template <bool EACH>
__device__ __forceinline__ void commit_class(const CommitParams& p, uint32_t class_mask, bool bump, bool active, int lane, const RingState* ahead = nullptr) {
  DevState* st = p.st;
  const int c = !EACH || active ? __ffs(class_mask) - 1 : 0;
  uint32_t* h = reinterpret_cast<uint32_t*>(p.hist + (size_t)c * p.H);
  const uint32_t H = p.H;
  uint32_t cnt = 0, newest = 0, m = 0, pos = 0;
  bool scan = false;
  if (!EACH || active) {
    newest = p.amax_override ? (__float_as_uint(__ldcg(p.amax_override)) & 0x7fffffffu) : __ldcg(&st->pending_amax[c]);
    const RingState now = ahead ? *ahead : ring_state(p, c);
    const uint32_t wmax = now.wmax, evicted = now.evicted;
    cnt = now.count;
    pos = cnt % H;
    m = newest >= wmax ? newest : wmax;
    scan = newest < wmax && evicted >= wmax;  // the maximum leaves: scan what stays
  }
  if (!EACH) {
    if (scan) m = max(newest, ring_max(h, H, pos, lane));
  } else {
    for (uint32_t left = __ballot_sync(0xffffffffu, scan); left; left &= left - 1) {
      const int who = __ffs(left) - 1;
      const uint32_t* ring = reinterpret_cast<const uint32_t*>(__shfl_sync(0xffffffffu, (unsigned long long)h, who));
      const uint32_t top = ring_max(ring, __shfl_sync(0xffffffffu, H, who), __shfl_sync(0xffffffffu, pos, who), lane);
      if (lane == who) m = max(newest, top);
    }
  }
  if (EACH ? active : lane == 0) {
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
    if (bump) atomicAdd(&st->token, 1ull);
  }
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
