// Sums between the blocks of one persistent solve on a cooperative grid,
// through tagged words in L2.
//
// What bounds one: the round trips to L2 that lie on the critical path
// (about 370 cycles each, 840 for a fence behind a store).  An arrival
// counter followed by a read of the partial sums takes the partials' fence,
// the atomic add, the poll that sees it and the read of the partials, and the
// adds of all blocks queue on one address.  Here every block publishes its
// partial sum and the sum's number in one 16-byte word of its own, so that
// the value arrives with the poll that sees the tag; blocks form groups of
// about sqrt(grid), the first of each adds its group's partials and publishes
// the group's sum the same way, and every block polls the groups' sums only
// (152 blocks polling all 152 words kept the words' own stores waiting: 9,600
// cycles a sum against 3,700 on 8 blocks).  The status word is read by one
// more lane in the same poll.
#pragma once

#include "dev_common.cuh"

namespace mmd {

__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ unsigned ld_relaxed(const unsigned* p) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// 16-byte {value, tag} words, read and written as one access
__device__ __forceinline__ void ld_tagged(const ulonglong2* p, unsigned long long& v, unsigned long long& tag) {
  asm volatile(
      "{\n .reg .b128 t;\n ld.relaxed.gpu.global.b128 t, [%2];\n mov.b128 {%0, %1}, t;\n}"
      : "=l"(v), "=l"(tag)
      : "l"(p)
      : "memory");
}
__device__ __forceinline__ void st_tagged(ulonglong2* p, unsigned long long v, unsigned long long tag) {
  asm volatile("{\n .reg .b128 t;\n mov.b128 t, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], t;\n}" ::"l"(p), "l"(v),
               "l"(tag)
               : "memory");
}

// One per block: the number of sums formed, and a failed wait (sticky).
struct CommSh {
  unsigned nred;
  int fail;
};

__device__ __forceinline__ void comm_init(CommSh& cs) {
  if (threadIdx.x == 0) {
    cs.nred = 0;
    cs.fail = 0;
  }
  __syncthreads();
}

// The value of one word once it carries `want`, by the calling thread alone;
// false when another block's status or the time limit ended the wait.
__device__ __forceinline__ bool wait_tagged(const GridBarrier& b, const ulonglong2* p, unsigned long long want,
                                            unsigned long long& v) {
  unsigned long long tg;
  ld_tagged(p, v, tg);
  if (tg == want) return true;
  const long long t0 = global_ns();
  for (unsigned spins = 0;; ++spins) {
    ld_tagged(p, v, tg);
    if (tg == want) return true;
    if ((spins & 31u) == 0u) {
      if (ld_relaxed((const unsigned*)b.status) != (unsigned)DEV_OK) return false;
      if (global_ns() - t0 > b.timeout_ns) {
        atomicCAS(b.status, (int)DEV_OK, (int)DEV_TIMEOUT);
        return false;
      }
    }
  }
}

// One poll round's verdict for the calling warp: 0 go on, 1 done, 2 give up
// (another block's status, or this wait's time limit).
__device__ __forceinline__ int poll_verdict(const GridBarrier& b, bool ready, unsigned status, unsigned& spins,
                                            long long t0) {
  if (__any_sync(0xffffffffu, status != (unsigned)DEV_OK)) return 2;
  if (__all_sync(0xffffffffu, ready)) return 1;
  if (((++spins) & 63u) == 1u) {
    const bool late = global_ns() - t0 > b.timeout_ns;
    if (__any_sync(0xffffffffu, late)) {
      if ((threadIdx.x & 31) == 0) atomicCAS(b.status, (int)DEV_OK, (int)DEV_TIMEOUT);
      return 2;
    }
  }
  return 0;
}

// Block-level sum of nv values: part[v * stride + t] is thread t's share,
// t < lim (the others hold nothing).  Every thread has stored its shares; the
// sums end in quart[v * 4 + q], q < wpc (returned).  An FP64 warp instruction
// occupies its sub-partition for 64 to 76 cycles however many lanes work, so
// a value's adds go to as few warps as keep the four sub-partitions busy (the
// shuffle tree costs a warp five): two for two values, one from three on.
__device__ __forceinline__ int block_sums(const double* part, int stride, int nv, int lim, double* quart) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wpc = lim <= 64 ? 1 : (nv <= 1 ? 4 : (nv <= 2 ? 2 : 1));
  __syncthreads();
  if (w < nv * wpc) {
    const int v = w / wpc, q = w - v * wpc;
    const double* p = part + v * stride;
    double t = 0.0;
    for (int i = q * 32 + lane; i < lim; i += 32 * wpc) t += p[i];
    t = warp_sum(t);
    if (lane == 0) quart[v * 4 + q] = t;
  }
  __syncthreads();
  return wpc;
}

// Sum of the n <= 32 words sl[0, n) once all carry `tag`, by one warp, in a
// fixed order; false when the wait was given up.
__device__ __forceinline__ bool poll_sum(const GridBarrier& b, const ulonglong2* sl, unsigned n, unsigned tag,
                                         double* sum) {
  const unsigned lane = threadIdx.x & 31;
  const long long t0 = global_ns();
  unsigned spins = 0;
  unsigned long long v;
  int verdict;
  do {
    unsigned long long tg = tag;
    unsigned st = DEV_OK;
    v = 0ull;
    if (lane < n) ld_tagged(sl + lane, v, tg);
    if (spins && lane == 0) st = ld_relaxed((const unsigned*)b.status);
    verdict = poll_verdict(b, tg == tag, st, spins, t0);
  } while (verdict == 0);
  double t = __longlong_as_double((long long)v);
  for (unsigned o = 16; o > 0; o >>= 1)
    if (o < n) t += __shfl_xor_sync(0xffffffffu, t, o);
  *sum = t;
  return verdict == 1;
}

// Blocks per group of a grid-wide sum: one level up to 16 blocks, else about
// sqrt(G); at most 32 groups of at most 32 blocks, so G <= 1024.
__host__ __device__ inline unsigned sum_group(unsigned G) {
  if (G <= 16) return 1;
  unsigned g = 4;
  while (g * g < G) ++g;
  return g;
}
// 16-byte words of the tagged sums of nvmax values on G blocks
__host__ __device__ inline size_t sum_words(int nvmax, unsigned G) { return size_t(2) * nvmax * (G + 32); }

// Largest grid whose fenced sums go through tagged words.
constexpr int kTaggedBlocks = 16;

// Grid-wide sums dst[v] (shared) of nv values in every block, all blocks
// adding the same partials in the same order.  FENCE: also a full barrier
// (what any thread wrote before it is seen after it), on at most
// kTaggedBlocks blocks, each of which reads every other's word; without, only
// the sums are exchanged, and a block has read everything it reads before it.
// b.slots: sum_words(nvmax, G) zeroed words; a block overwrites the words of
// sum R with those of sum R + 2, after every block has published sum R + 1
// and so has read sum R.  blockDim >= 32 nv.
template <bool FENCE>
__device__ __forceinline__ bool grid_sums(const GridBarrier& b, CommSh& cs, const double* part, int stride, int nv,
                                          int nvmax, int lim, double* quart, double* dst) {
  const int wpc = block_sums(part, stride, nv, lim, quart);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned G = gridDim.x, gs = FENCE ? 1 : sum_group(G);
  const unsigned tag = cs.nred + 1;
  if (w < nv) {
    ulonglong2* sl = b.slots + (size_t(tag & 1u) * nvmax + w) * (G + 32);
    if (lane == 0) {
      double t = quart[w * 4];
      for (int q = 1; q < wpc; ++q) t += quart[w * 4 + q];
      if (FENCE) fence_gpu();
      st_tagged(sl + blockIdx.x, (unsigned long long)__double_as_longlong(t), tag);
    }
    bool ok = true;
    double t = 0.0;
    if (gs == 1) {
      ok = poll_sum(b, sl, G, tag, &t);
    } else {
      if (blockIdx.x % gs == 0) {  // first of its group
        ok = poll_sum(b, sl + blockIdx.x, min(gs, G - blockIdx.x), tag, &t);
        if (ok && lane == 0)
          st_tagged(sl + G + blockIdx.x / gs, (unsigned long long)__double_as_longlong(t), tag);
      }
      if (ok) ok = poll_sum(b, sl + G, (G + gs - 1) / gs, tag, &t);
    }
    if (lane == 0) {
      dst[w] = t;
      if (!ok) cs.fail = 1;
    }
    if (FENCE) fence_gpu();
  }
  __syncthreads();
  if (threadIdx.x == 0) cs.nred = tag;
  return cs.fail == 0;
}

}  // namespace mmd
