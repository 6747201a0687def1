// CG on A (mode 0 of the persistent solver, FP64) with every row owned by one
// thread for the whole solve.
//
// The recurrence is Chronopoulos-Gear CG: w = A r with r^T r and r^T w in one
// pass, one grid-wide sum, then p = r + beta p, s = w + beta s, x += alpha p,
// r -= alpha s in a second pass.  A lane keeps the rows of its SELL slices
// through both passes, so p, s, x, w and its own r never leave the SM's
// shared memory, and only r crosses SMs.
//
// What bounds an iteration: the latency of the exchange at small sizes, the
// FP64 unit (one warp instruction per 19 cycles and SM, whatever the lanes)
// at large ones, and the rate of the scattered gathers, about two cycles a
// word through L1 whether they hit or not.  So the rows that a block's entries
// read are listed once per matrix and grid (near_kernel), every iteration
// copies their r into shared memory, each row once and in row order, and the
// entries gather from there by 16-bit local indices.  r is stored as {value,
// tag} words, so that this copy is the barrier too: it waits for the values
// themselves.  The block's part of the matrix is staged in shared memory, as
// many slices as fit, the rest is streamed from L2.
//
// Measured, us an iteration, solve_kernel on the rows as they came -> here:
// 64 x 64 operator 9.7 -> 4.6, 256 x 256 12.0 -> 6.7; 10-nearest-neighbour
// graphs of 2k rows 10.5 -> 5.3, 20k 14.5 -> 7.1, 50k 15.5 -> 8.2, 200k 20.5 ->
// 15.3 (17.8 before in the order of a handle's patches); geometric graph of 100k
// rows 16.0 -> 9.2.  Where it would lose: own_plan.
//
// Two instances:
//   grid     a cooperative launch over many SMs, sums and barriers of
//            grid_comm.cuh;
//   cluster  the whole problem in one thread-block cluster of up to 16 SMs,
//            sums through distributed shared memory, the hardware cluster
//            barrier.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "grid_comm.cuh"
#include "kernels.h"

namespace mmd {

namespace {

constexpr int kOwnVecs = 5;          // w, r, p, s, x
// Threads of a block.  One warp per SM sub-partition already issues FP64 at
// the unit's rate (one warp instruction per 19 cycles and SM), so more warps
// only cover load latency, and cost: a block barrier takes about 600 cycles
// at 1024 threads, and every thread's share of a sum is one more FP64 add.
constexpr int kOwnThreads = 256;
constexpr int kOwnUnits = 24;  // most parts of split slices
constexpr int kOwnMaxCluster = 16;

struct OwnSh {
  CommSh comm;
  double quart[2 * 4];
  double sum[2];  // of one reduction: delta, gamma (set-up: b^T b, r^T r)
  double bn, irz, den, alpha, beta;
  int act;
  long long it;
  double box[2][2][kOwnMaxCluster];  // cluster: every block's partial sums
  int late[2][kOwnMaxCluster];       // cluster: a block's wait ran over its limit
};

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned map_rank(unsigned addr, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster(unsigned addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ void st_cluster_int(unsigned addr, int v) {
  asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

extern __shared__ double g_own[];

// The rows that the entries of block b's slices read, ascending, into
// list[b stride ..], their number into count[b] (stride + 1 where they are
// more than stride, and nothing is listed), and every entry's place in that
// list into lcol (SELL order).  A bit per row of the matrix in shared memory;
// the rank of a bit is its word's prefix count plus the bits below it.
__global__ void near_kernel(Sell A, int64_t n, const int32_t* first, int stride, int32_t* count, int32_t* list,
                            uint16_t* lcol) {
  __shared__ int s_tot[32];
  unsigned* bits = (unsigned*)g_own;
  const int words = (int)((n + 31) >> 5), tid = threadIdx.x, NT = blockDim.x, lane = tid & 31, w = tid >> 5;
  int* rank = (int*)bits + words;
  const int32_t e0 = A.ptr[first[blockIdx.x]], e1 = A.ptr[first[blockIdx.x + 1]];
  for (int i = tid; i < words; i += NT) bits[i] = 0u;
  __syncthreads();
  for (int32_t e = e0 + tid; e < e1; e += NT) atomicOr(bits + (A.col[e] >> 5), 1u << (A.col[e] & 31));
  __syncthreads();
  int H = 0;
  for (int base = 0; base < words; base += NT) {
    const int i = base + tid;
    const int v = i < words ? __popc(bits[i]) : 0;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    if (lane == 31) s_tot[w] = inc;
    __syncthreads();
    int before = 0, all = 0;
    for (int q = 0; q < (NT >> 5); ++q) {
      if (q < w) before += s_tot[q];
      all += s_tot[q];
    }
    if (i < words) rank[i] = H + before + inc - v;
    H += all;
    __syncthreads();
  }
  if (tid == 0) count[blockIdx.x] = H <= stride ? H : stride + 1;
  if (H > stride) return;
  int32_t* out = list + size_t(blockIdx.x) * stride;
  for (int i = tid; i < words; i += NT) {
    int at = rank[i];
    for (unsigned u = bits[i]; u; u &= u - 1) out[at++] = i * 32 + __ffs(u) - 1;
  }
  for (int32_t e = e0 + tid; e < e1; e += NT) {
    const int32_t j = A.col[e];
    lcol[e] = (uint16_t)(rank[j >> 5] + __popc(bits[j >> 5] & ((1u << (j & 31)) - 1u)));
  }
}

// Sums over the cluster: every block stores its partials into every block's
// box, one hardware barrier, and each block adds them in rank order.
__device__ __forceinline__ bool cluster_sums(const GridBarrier& b, OwnSh& s, const double* part, int stride, int lim) {
  constexpr int nv = 2;
  const int wpc = block_sums(part, stride, nv, lim, s.quart);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int C = gridDim.x, me = (int)cluster_rank();
  const unsigned tag = s.comm.nred + 1, par = tag & 1u;
  for (int t = threadIdx.x; t < nv * C; t += blockDim.x) {
    const int v = t / C, to = t - v * C;
    double q = s.quart[v * 4];
    for (int i = 1; i < wpc; ++i) q += s.quart[v * 4 + i];
    st_cluster(map_rank(smem_addr(&s.box[par][v][me]), to), q);
    if (v == 0) st_cluster_int(map_rank(smem_addr(&s.late[par][me]), to), s.comm.fail);
  }
  const long long t0 = global_ns();
  cluster_barrier();
  const bool over = global_ns() - t0 > b.timeout_ns;
  if (w < nv) {
    double t = lane < C ? s.box[par][w][lane] : 0.0;
    for (int o = 8; o > 0; o >>= 1)
      if (o < C) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) s.sum[w] = t;
  }
  int late = 0;
  for (int i = 0; i < C; ++i) late |= s.late[par][i];
  __syncthreads();
  if (threadIdx.x == 0) {
    s.comm.nred = tag;
    // told to the other blocks with the next sums, so that all leave together
    if (over) {
      s.comm.fail = 1;
      atomicCAS(b.status, (int)DEV_OK, (int)DEV_TIMEOUT);
    }
  }
  return late == 0;
}

template <bool CL>
__global__ void __launch_bounds__(kOwnThreads, 1) own_cg_kernel(SolverArgs a, OwnPlan pl) {
  __shared__ OwnSh s;
  comm_init(s.comm);
  // a block's shared memory may be written by its peers once it runs: the first sums store into it
  if constexpr (CL) cluster_barrier();
  constexpr int NT = kOwnThreads, nw = NT / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const Sell& A = a.A;
  const int64_t lo = pl.first[blockIdx.x], hi = pl.first[blockIdx.x + 1];
  const int nsl = (int)(hi - lo), S = pl.slots;  // S: slots (32 per slice) of the largest share
  const int lim = min(NT, nsl * 32);
  const double* __restrict__ b = (const double*)a.b;
  double* __restrict__ x = (double*)a.x;
  // r crosses SMs as {value, tag} words: a block's copy of its listed rows waits for each value
  // itself, and no barrier stands between the update and the next product
  ulonglong2* const rt = pl.rt;
  const unsigned long long epoch = (unsigned long long)pl.epoch << 32;
  // ---- dynamic shared memory
  double* const part = g_own;                  // 2 x NT: the threads' shares of a sum
  double* const comb = part + 2 * NT;          // sums of the parts of split slices
  double* const wv = comb + kOwnUnits * 32;    // the owned vectors, S slots each
  double* const rv = wv + S;
  double* const pv = rv + S;
  double* const sv = pv + S;
  double* const xv = sv + S;
  int32_t* const srow = (int32_t*)(xv + S);    // row of each slot
  int2* const smeta = (int2*)(srow + S);       // per slice: first entry, width
  double* const near = (double*)(smeta + S / 32);
  int32_t* const list = (int32_t*)(near + pl.near);
  double* const sval = (double*)(list + pl.near);
  uint16_t* const scol = (uint16_t*)(sval + pl.ents);
  const int H = pl.count[blockIdx.x];
  const int32_t e0 = A.ptr[lo];
  int nst = 0;  // slices [0, nst) are staged
  while (nst < nsl && A.ptr[lo + nst + 1] - e0 <= pl.ents) ++nst;
  for (int i = tid; i < H; i += NT) list[i] = pl.list[size_t(blockIdx.x) * pl.stride + i];
  {
    const int32_t ents = A.ptr[lo + nst] - e0;
    for (int e = tid; e < ents; e += NT) {
      sval[e] = A.val[e0 + e];
      scol[e] = pl.lcol[e0 + e];
    }
  }
  for (int q = tid; q < nsl * 32; q += NT) srow[q] = A.row[lo * 32 + q];
  for (int q = tid; q < nsl; q += NT) smeta[q] = make_int2(A.ptr[lo + q], A.len[lo + q]);
  __syncthreads();

  auto sums = [&]() -> bool {  // the two values in part -> s.sum, in every block
    if constexpr (CL)
      return cluster_sums(a.bar, s, part, NT, lim);
    else
      return grid_sums<false>(a.bar, s.comm, part, NT, 2, 2, lim, s.quart, s.sum);
  };

  // ---- set-up: r = b - A x0 (or b); sums of b^2 and r^2
  double acc = 0.0, acc2 = 0.0;
  for (int sl = warp; sl < nsl; sl += nw) {
    const int q = sl * 32 + lane;
    const int32_t row = srow[q];
    double ax = 0.0;
    if (a.x0) {
      const int32_t g0 = smeta[sl].x + lane, len = smeta[sl].y;
      for (int k = 0; k < len; ++k) ax = fma(A.val[g0 + k * 32], x[A.col[g0 + k * 32]], ax);
    }
    const double bv = row >= 0 ? b[row] : 0.0;
    const double r0 = row >= 0 ? bv - ax : 0.0;
    xv[q] = (a.x0 && row >= 0) ? x[row] : 0.0;
    rv[q] = r0;
    if (row >= 0) st_tagged(rt + row, (unsigned long long)__double_as_longlong(r0), epoch);
    acc = fma(bv, bv, acc);
    acc2 = fma(r0, r0, acc2);
  }
  part[tid] = acc;
  part[NT + tid] = acc2;
  if (!sums()) return;
  if (tid == 0) {
    s.bn = s.sum[0];
    s.act = (s.bn > 0.0) && !(sqrt(s.sum[1]) <= a.tol * sqrt(s.bn));
    s.it = 0;
  }
  __syncthreads();

  for (int it = 1; s.act; ++it) {
    // the listed rows' r of the last update: a thread waits for its first word, the others have
    // mostly come by then and are read at once
    {
      const unsigned long long want = epoch | (unsigned)(it - 1);
      constexpr int UN = 8;
      bool ok = true;
      for (int i0 = tid; i0 < H && ok; i0 += UN * NT) {
        unsigned long long v[UN], tg[UN];
        ok = wait_tagged(a.bar, rt + list[i0], want, v[0]);
#pragma unroll
        for (int u = 1; u < UN; ++u) {
          tg[u] = want;
          if (i0 + u * NT < H) ld_tagged(rt + list[i0 + u * NT], v[u], tg[u]);
        }
        near[i0] = __longlong_as_double((long long)v[0]);
#pragma unroll
        for (int u = 1; u < UN; ++u)
          if (i0 + u * NT < H) {
            if (tg[u] != want) ok = wait_tagged(a.bar, rt + list[i0 + u * NT], want, v[u]) && ok;
            near[i0 + u * NT] = __longlong_as_double((long long)v[u]);
          }
      }
      if (!ok) s.comm.fail = 1;
    }
    __syncthreads();
    if (!CL && s.comm.fail) return;  // a cluster's blocks are told with the next sums
    // w = A r; delta = r^T w, gamma = r^T r.  A small share waits for the FMA chains of its widest
    // rows: a slice's entries are dealt to several warps then, and their sums added afterwards (a
    // barrier and the adds, about 400 cycles, against 85 an entry: parts of eight entries at
    // least).  Up to kOwnUnits parts in all, three rounds of the warps; from 13 slices on the
    // chains overlap anyway.
    acc = acc2 = 0.0;
    int parts = 1;
    while (parts < 8 && nsl * parts * 2 <= kOwnUnits && smeta[0].y >= 16 * parts) parts *= 2;
    auto row_done = [&](int q, double ax) {
      const double r0 = rv[q];
      wv[q] = ax;
      acc = fma(r0, ax, acc);
      acc2 = fma(r0, r0, acc2);
    };
    for (int un = warp; un < nsl * parts; un += nw) {
      const int sl = un / parts, pt = un - sl * parts;
      const int2 mt = smeta[sl];
      const int k0 = mt.y * pt / parts, len = mt.y * (pt + 1) / parts - k0;
      double ax = 0.0;
      if (len <= 0) {
      } else if (sl < nst) {
        // staged: an entry's value and place are read two entries ahead of its FMA, its r one
        // ahead (past the end the last entry again); 85 cycles an entry for one warp, the FP64
        // rate from two warps per sub-partition on
        const double* av = sval + (mt.x - e0) + k0 * 32 + lane;
        const uint16_t* jv = scol + (mt.x - e0) + k0 * 32 + lane;
        const int o1 = min(1, len - 1) * 32;
        double e = av[0], g = near[jv[0]], en = av[o1];
        int jn = jv[o1];
#pragma unroll 4
        for (int k = 0; k < len; ++k) {
          const double gn = near[jn];
          const int o2 = min(k + 2, len - 1) * 32;
          const double e2 = av[o2];
          const int j2 = jv[o2];
          ax = fma(e, g, ax);
          e = en;
          g = gn;
          en = e2;
          jn = j2;
        }
      } else {
        // streamed from L2: eight entries ahead
        constexpr int UE = 8;
        const double* __restrict__ av = A.val + mt.x + k0 * 32 + lane;
        const uint16_t* __restrict__ jv = pl.lcol + mt.x + k0 * 32 + lane;
        double e[UE];
        int j[UE];
#pragma unroll
        for (int u = 0; u < UE; ++u) {
          const int o = min(u, len - 1) * 32;
          e[u] = __ldg(av + o);
          j[u] = __ldg(jv + o);
        }
        for (int k = 0; k < len; k += UE) {
#pragma unroll
          for (int u = 0; u < UE; ++u) {
            const double g = near[j[u]], f = e[u];
            const int o = min(k + UE + u, len - 1) * 32;
            e[u] = __ldg(av + o);
            j[u] = __ldg(jv + o);
            if (k + u < len) ax = fma(f, g, ax);
          }
        }
      }
      if (parts > 1)
        comb[un * 32 + lane] = ax;
      else if (srow[sl * 32 + lane] >= 0)
        row_done(sl * 32 + lane, ax);
    }
    if (parts > 1) {
      __syncthreads();
      for (int sl = warp; sl < nsl; sl += nw) {
        const int q = sl * 32 + lane;
        if (srow[q] < 0) continue;
        double ax = comb[sl * parts * 32 + lane];
        for (int p = 1; p < parts; ++p) ax += comb[(sl * parts + p) * 32 + lane];
        row_done(q, ax);
      }
    }
    if (tid < lim) {
      part[tid] = acc;
      part[NT + tid] = acc2;
    }
    if (!sums()) return;
    if (tid == 0) {
      const double dl = s.sum[0], g = s.sum[1];
      if (it > 1 && g <= a.tol * a.tol * s.bn) {
        s.act = 0;  // converged after update it - 1
      } else if (it <= a.maxit) {
        // beta = gamma / gamma', alpha = gamma / (delta - beta gamma / alpha'); with
        // alpha' = gamma' / den' the subtracted term is beta^2 den': one division on the path
        double be = 0.0, den = dl;
        if (it > 1) {
          be = g * s.irz;
          den = fma(-be * be, s.den, dl);
        }
        if (!(den > 0.0)) {
          s.act = 0;
          if (blockIdx.x == 0) atomicExch(a.bar.status, (int)DEV_NOTSPD);
        }
        s.den = den;
        s.alpha = g / den;
        s.beta = be;
        s.it = it;
      }
    }
    __syncthreads();
    if (it > a.maxit || !s.act) break;  // still active at the cap: reports no convergence
    if (tid == NT - 1) s.irz = 1.0 / s.sum[1];  // next iteration's 1 / gamma'
    // p = r + beta p, s = w + beta s, x += alpha p, r -= alpha s
    const bool first = (it == 1);
    const double be = s.beta, al = s.alpha;
    for (int sl = warp; sl < nsl; sl += nw) {
      const int q = sl * 32 + lane;
      const int32_t row = srow[q];
      if (row < 0) continue;
      const double r0 = rv[q], w0 = wv[q];
      const double sn = first ? w0 : fma(be, sv[q], w0);
      const double rn = fma(-al, sn, r0);
      st_tagged(rt + row, (unsigned long long)__double_as_longlong(rn), epoch | (unsigned)it);
      const double pn = first ? r0 : fma(be, pv[q], r0);
      rv[q] = rn;
      pv[q] = pn;
      sv[q] = sn;
      xv[q] = fma(al, pn, xv[q]);
    }
  }
  for (int sl = warp; sl < nsl; sl += nw) {
    const int q = sl * 32 + lane;
    const int32_t row = srow[q];
    if (row >= 0) x[row] = s.bn == 0.0 ? 0.0 : xv[q];  // a zero right-hand side gives x = 0
  }
  if (blockIdx.x == 0 && tid == 0) {
    a.it_out[0] = s.it;
    a.conv[0] = s.act ? 0 : 1;
  }
}

int current_device() {
  int d = -1;
  return cudaGetDevice(&d) == cudaSuccess ? d : -1;
}

template <bool CL>
void own_attrs() {
  static PerDevice once;
  once.run(current_device(), [] {
    cudaFuncSetAttribute(own_cg_kernel<CL>, cudaFuncAttributeMaxDynamicSharedMemorySize, kOwnSmem);
    if (CL) cudaFuncSetAttribute(own_cg_kernel<CL>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  });
}

}  // namespace

// Blocks that may list their rows: a bit and a count per 32 rows in shared memory.
bool near_fits(int64_t n) { return ((n + 31) / 32) * 8 <= kOwnSmem; }

cudaError_t launch_near(const Sell& A, int64_t n, int grid, const int32_t* first, int stride, int32_t* count,
                        int32_t* list, uint16_t* lcol, cudaStream_t st) {
  static PerDevice once;
  once.run(current_device(), [] {
    cudaFuncSetAttribute(near_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kOwnSmem);
  });
  near_kernel<<<grid, 1024, ((n + 31) / 32) * 8, st>>>(A, n, first, stride, count, list, lcol);
  return cudaGetLastError();
}

// Block b of a launch takes the slices [first[b], first[b + 1]): shares of
// equal work, a slice costing its entries' FMAs and six more (two dot
// products, four updates).  Equal numbers of slices left blocks waiting: a
// window's slices are sorted by width.
std::vector<int32_t> own_shares(const int32_t* sptr, int64_t nslices, int grid) {
  std::vector<int32_t> first(grid + 1, (int32_t)nslices);
  const double total = sptr[nslices] / 32.0 + 6.0 * nslices;
  int64_t sl = 0;
  for (int b = 0; b < grid; ++b) {
    const double goal = total * b / grid;
    while (sl < nslices && (int64_t(sptr[sl]) + sptr[sl + 1]) / 64.0 + 6.0 * sl + 3.0 < goal) ++sl;  // nearest boundary
    first[b] = (int32_t)sl;
  }
  first[0] = 0;
  return first;
}

bool own_plan(const int32_t* sptr, const int32_t* first, int grid, int near, OwnPlan* out) {
  OwnPlan p;
  int64_t ents = 0, slices = 0;
  for (int b = 0; b < grid; ++b) {
    ents = std::max<int64_t>(ents, sptr[first[b + 1]] - sptr[first[b]]);
    slices = std::max<int64_t>(slices, first[b + 1] - first[b]);
  }
  if (slices < 1 || near < 1) return false;
  p.near = (near + 1) & ~1;  // what follows starts on 8 bytes
  const int64_t used = int64_t(8) * (2 * kOwnThreads + kOwnUnits * 32) +
                       slices * (32 * (8 * kOwnVecs + 4) + int64_t(sizeof(int2))) + int64_t(12) * p.near;
  if (used > kOwnSmem) return false;
  p.slots = (int)slices * 32;
  p.ents = (int)(std::min<int64_t>((kOwnSmem - used) / 10, ents) & ~int64_t(31));  // slices hold multiples of 32
  if (p.ents < ents && 10 * p.ents < kOwnStaged) return false;
  if (4 * int64_t(near) > 3 * ents && 4 * int64_t(p.ents) < 3 * ents) return false;
  p.smem = (int)(used + int64_t(10) * p.ents);
  *out = p;
  return true;
}

template <bool CL>
static cudaLaunchConfig_t own_config(int grid, int smem, cudaStream_t st, cudaLaunchAttribute* at) {
  own_attrs<CL>();
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kOwnThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  if (CL) {
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = grid;
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
  } else {
    at->id = cudaLaunchAttributeCooperative;
    at->val.cooperative = 1;
  }
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

bool own_cluster_fits(int ranks) {
  cudaLaunchAttribute at;
  const cudaLaunchConfig_t cfg = own_config<true>(ranks, kOwnSmem, nullptr, &at);
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, own_cg_kernel<true>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return n >= 1;
}

int own_max_grid(int num_sms) {
  own_attrs<false>();
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, own_cg_kernel<false>, kOwnThreads, kOwnSmem);
  return nb >= 1 ? std::min(num_sms, 1024) : 0;
}

cudaError_t launch_own_cg(const SolverArgs& a, const OwnPlan& p, int grid, bool cluster, cudaStream_t st) {
  if (a.mode != 0 || a.fp32 || a.df || a.b64 || a.m != 1 || grid < 1) return cudaErrorInvalidValue;
  if (cluster && grid > kOwnMaxCluster) return cudaErrorInvalidValue;
  cudaLaunchAttribute at;
  if (cluster) {
    const cudaLaunchConfig_t cfg = own_config<true>(grid, p.smem, st, &at);
    return cudaLaunchKernelEx(&cfg, own_cg_kernel<true>, a, p);
  }
  const cudaLaunchConfig_t cfg = own_config<false>(grid, p.smem, st, &at);
  return cudaLaunchKernelEx(&cfg, own_cg_kernel<false>, a, p);
}

}  // namespace mmd
