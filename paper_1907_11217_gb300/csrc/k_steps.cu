// Per-group kernels: leaf builder, direct small-step contraction, FP64
// accumulation of partial amplitudes.
#include <algorithm>
#include <mutex>

#include "kernels.h"

namespace tz {
namespace dev {

// complex arithmetic on float2 (complex64) and double2 (complex128)
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cfma(float2 a, float2 b, float2 c) {
  c.x = fmaf(a.x, b.x, c.x);
  c.x = fmaf(-a.y, b.y, c.x);
  c.y = fmaf(a.x, b.y, c.y);
  c.y = fmaf(a.y, b.x, c.y);
  return c;
}
__device__ __forceinline__ double2 cfma(double2 a, double2 b, double2 c) {
  c.x = fma(a.x, b.x, c.x);
  c.x = fma(-a.y, b.y, c.x);
  c.y = fma(a.x, b.y, c.y);
  c.y = fma(a.y, b.x, c.y);
  return c;
}
template <typename T>
__device__ __forceinline__ T czero();
template <>
__device__ __forceinline__ float2 czero<float2>() { return make_float2(0.f, 0.f); }
template <>
__device__ __forceinline__ double2 czero<double2>() { return make_double2(0.0, 0.0); }
__device__ __forceinline__ float2 table_value(const LeafJob &j, int i, float2 *) { return j.M[i]; }
__device__ __forceinline__ double2 table_value(const LeafJob &j, int i, double2 *) { return j.Md[i]; }

// Starts a call: the group state, and with n_acc > 0 the accumulator cleared
// (one launch instead of a memset and a launch).
__global__ void init_state_kernel(GroupState *gs, int64_t lo, int64_t hi, int64_t n_rows, int keep_error, double2 *acc,
                                  int64_t n_acc) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_acc; i += (int64_t)gridDim.x * blockDim.x)
    acc[i] = make_double2(0.0, 0.0);
  if (blockIdx.x != 0 || threadIdx.x != 0) return;
  gs->slice = lo;
  gs->chunk = 0;
  gs->lo = lo;
  gs->hi = hi;
  gs->n_rows = n_rows;
  gs->groups_done = 0;
  if (!keep_error) gs->tc_error = 0;
}

cudaError_t launch_init_state(GroupState *gs, int64_t lo, int64_t hi, int64_t n_rows, double2 *acc, int64_t n_acc,
                              cudaStream_t s, int keep_error) {
  const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((n_acc + 255) / 256, 152 * 8));
  init_state_kernel<<<(unsigned)blocks, 256, 0, s>>>(gs, lo, hi, n_rows, keep_error, acc, n_acc);
  return cudaGetLastError();
}

// One block per leaf job. Gather: a constant tensor with its sliced bits
// fixed to the bits of the current slice id (Sec. 1 subtasks). Output: the
// tensor <x_q| (final gates folded in) for the current chunk of bitstrings.
template <typename T>
__global__ void leaf_kernel(const LeafJob *jobs, const GroupState *gs, const uint8_t *bits, int nq, int g,
                            const char *cbase, char *abase) {
  // the block's job, staged with one round of loads (field by field they
  // depend on one another)
  static_assert(sizeof(LeafJob) % 16 == 0 && sizeof(LeafJob) / 16 <= 128, "LeafJob staged by 128 threads");
  __shared__ __align__(16) char s_job[sizeof(LeafJob)];
  if (threadIdx.x < sizeof(LeafJob) / 16)
    reinterpret_cast<uint4 *>(s_job)[threadIdx.x] = reinterpret_cast<const uint4 *>(jobs + blockIdx.x)[threadIdx.x];
  const int64_t slice = gs->slice, chunk = gs->chunk, n_rows = gs->n_rows;
  __syncthreads();
  const LeafJob &j = *reinterpret_cast<const LeafJob *>(s_job);
  T *dst = const_cast<T *>(region_ptr<T>(j.dst, cbase, abase));
  const T *src = j.kind == LJ_GATHER ? region_ptr<T>(j.src, cbase, abase) : nullptr;
  const int64_t n = int64_t(1) << j.rank;
  for (int64_t e = threadIdx.x; e < n; e += blockDim.x) {
    if (j.kind == LJ_GATHER) {
      int64_t so = 0;
      for (int p = 0; p < j.rank; p++) so |= ((e >> p) & 1) << j.src_pos[p];
      for (int f = 0; f < j.n_fixed; f++) so |= ((slice >> j.fixed_slice_bit[f]) & 1) << j.fixed_src_pos[f];
      dst[e] = src[so];
    } else {
      int64_t beta = 0;
      for (int b = 0; b < g; b++)
        if (j.beta_dst_pos[b] >= 0) beta |= ((e >> j.beta_dst_pos[b]) & 1) << b;
      const int64_t row = (chunk << g) | beta;
      const int x = row < n_rows ? (bits[row * nq + j.qubit] & 1) : 0;
      int ev = 0;
      if (j.rc) {
        if (j.e_dst_pos >= 0)
          ev = (int)((e >> j.e_dst_pos) & 1);
        else if (j.e_slice_bit >= 0)
          ev = (int)((slice >> j.e_slice_bit) & 1);
      }
      dst[e] = table_value(j, x * (1 << j.rc) + ev, (T *)nullptr);
    }
  }
}

cudaError_t launch_leaf_build(const LeafJob *jobs, int n_jobs, const GroupState *gs, const uint8_t *bits, int nq,
                              int g, const char *cbase, char *abase, int dbl, cudaStream_t s) {
  if (dbl)
    leaf_kernel<double2><<<n_jobs, 128, 0, s>>>(jobs, gs, bits, nq, g, cbase, abase);
  else
    leaf_kernel<float2><<<n_jobs, 128, 0, s>>>(jobs, gs, bits, nq, g, cbase, abase);
  return cudaGetLastError();
}

__device__ __forceinline__ float2 shfl_c(float2 v, int l) {
  return make_float2(__shfl_sync(0xffffffffu, v.x, l), __shfl_sync(0xffffffffu, v.y, l));
}
__device__ __forceinline__ double2 shfl_c(double2 v, int l) {
  return make_double2(__shfl_sync(0xffffffffu, v.x, l), __shfl_sync(0xffffffffu, v.y, l));
}
// sum + v of lanes first .. first + n - 1, in order. The shuffles do not wait
// for one another, so this costs n additions in series (4 cycles each): about
// what a tree's few dependent shuffles cost, and the order of a plain loop.
template <typename T>
__device__ __forceinline__ T add_lanes(T sum, T v, int first, int n) {
#pragma unroll 4
  for (int q = 0; q < n; q++) {
    const T w = shfl_c(v, first + q);
    sum.x += w.x;
    sum.y += w.y;
  }
  return sum;
}
// Sum over the 2^split parts of an output that sit in consecutive lanes
// (split <= 5), in order.
template <typename T>
__device__ __forceinline__ T warp_parts(T v, int split) {
  if (split == 0) return v;
  const int first = (int)(threadIdx.x & 31) & ~((1 << split) - 1);
  return add_lanes(shfl_c(v, first), v, first + 1, (1 << split) - 1);
}

// One part of one output: the terms of its share of the summed bits, in
// Gray-code order (one offset update per term; a direct step touches at most
// 2^26 element combinations, so offsets fit 32 bits). L2: operands read
// through L2 (written earlier in the same launch by other SMs). The pointers
// are not __restrict__: in a chain the operands are other steps' results of
// the same launch, which a read-only load could miss.
template <typename T, bool L2>
__device__ __forceinline__ T direct_part(const DStep &st, uint32_t c, int part, const T *Ap, const T *Bp) {
  auto ld = [](const T *p) { return L2 ? __ldcg(p) : *p; };
  uint32_t oa = 0, ob = 0;
  for (int q = 0; q < st.nC; q++) {
    if (!((c >> q) & 1)) continue;
    if (st.a_c[q] >= 0) oa |= 1u << st.a_c[q];
    if (st.b_c[q] >= 0) ob |= 1u << st.b_c[q];
  }
  const int nlow = st.nK - st.split;
  for (int q = 0; q < st.split; q++)
    if ((part >> q) & 1) {
      oa |= 1u << st.a_k[nlow + q];
      ob |= 1u << st.b_k[nlow + q];
    }
  T acc = cmul(ld(Ap + oa), ld(Bp + ob));
  const uint32_t nt = 1u << nlow;
#pragma unroll 4
  for (uint32_t t = 1; t < nt; t++) {
    const int q = __ffs(t) - 1;
    oa ^= 1u << st.a_k[q];
    ob ^= 1u << st.b_k[q];
    acc = cfma(ld(Ap + oa), ld(Bp + ob), acc);
  }
  return acc;
}

// Direct contraction of small steps. Each output element is summed by
// 2^split consecutive threads, each walking its share of the contracted bits
// in Gray-code order (one offset update per term), then reduced. blk is the
// block's number within its step.
template <typename T>
__device__ __forceinline__ void direct_block(const DStep &st, int64_t blk, const char *cbase, char *abase, T *red) {
  const T *Ap = region_ptr<T>(st.A, cbase, abase);
  const T *Bp = region_ptr<T>(st.B, cbase, abase);
  T *Cp = const_cast<T *>(region_ptr<T>(st.C, cbase, abase));
  const int split = st.split;
  const int64_t item = blk * 256 + threadIdx.x;
  const int64_t c = item >> split;
  const int part = (int)(item & ((1 << split) - 1));
  const bool active = c < (int64_t(1) << st.nC);
  T acc = active ? direct_part<T, false>(st, (uint32_t)c, part, Ap, Bp) : czero<T>();
  if (split > 5) {  // 2, 4 or 8 warps an output
    red[threadIdx.x] = acc;
    __syncthreads();
    if (active && part == 0) {
      // (unrolled, so that the reads do not wait for the additions)
#pragma unroll 8
      for (int q = 1; q < (1 << split); q++) {
        const T v = red[threadIdx.x + q];
        acc.x += v.x;
        acc.y += v.y;
      }
    }
  } else {
    acc = warp_parts(acc, split);
  }
  if (active && part == 0) Cp[c] = acc;
}

// A block's step descriptor, staged in shared memory by 12 threads at once
// (its fields are then read by every thread without further global loads).
__device__ __forceinline__ void stage_step(DStep *dst, const DStep *src) {
  static_assert(sizeof(DStep) % 16 == 0 && sizeof(DStep) / 16 <= 32, "DStep staged in 16-byte pieces");
  if (threadIdx.x < sizeof(DStep) / 16)
    reinterpret_cast<uint4 *>(dst)[threadIdx.x] = reinterpret_cast<const uint4 *>(src)[threadIdx.x];
}

// One launch per dependency level: block b of the launch belongs to step
// bmap[b].
template <typename T>
__global__ void __launch_bounds__(256) direct_kernel(const DStep *steps, const int *bmap, const char *cbase,
                                                     char *abase) {
  __shared__ __align__(16) DStep s_st;
  __shared__ T red[256];
  const int64_t blk = blockIdx.x;
  stage_step(&s_st, steps + bmap[blk]);
  __syncthreads();
  direct_block<T>(s_st, blk - s_st.block_begin, cbase, abase, red);
}

cudaError_t launch_direct(const DStep *steps, int n_steps, const int *bmap, int64_t total_blocks, const char *cbase,
                          char *abase, int dbl, cudaStream_t s) {
  if (n_steps <= 0) return cudaSuccess;
  if (total_blocks > 0x7fffffffLL || !bmap) return cudaErrorInvalidValue;
  if (dbl)
    direct_kernel<double2><<<(unsigned)total_blocks, 256, 0, s>>>(steps, bmap, cbase, abase);
  else
    direct_kernel<float2><<<(unsigned)total_blocks, 256, 0, s>>>(steps, bmap, cbase, abase);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- chain
// A run of small dependency levels in one launch: one cluster of CTAs (at
// most eight) takes the levels one after the other, with a barrier of the
// cluster between them, where a launch per level is bound by launch latency
// (a replayed graph spends about 2.5 us a level, whose work takes under one).
// Work is dealt to warps, not blocks: small steps have a handful of outputs.
// A warp has at most one task in a level: 32 items of a step (output, part of
// the summed bits), a few terms each (the plan chains no other levels). Parts are
// added in the order of direct_block, so the results are bit-identical to it.
// A warp reads its task of the next level before the barrier. Operands are read
// through L2 where other CTAs wrote them a level before.
// Bound by latency (dependent loads and the barrier): a level takes about a
// microsecond less than its launch, and the chain 1 to 2 us to start. The
// twelve levels of at most 16 tasks of a 4 x 4 circuit of depth 10: 48.2 us a
// call as launches, 36.0 in a chain of one CTA (42.2 in a cluster of two with
// the level of 22 tasks before them).
// tab: n_levels pairs (first task, tasks), then the tasks (step, number
// within the step).
constexpr int kChainThreads = 512, kChainWarps = kChainThreads / 32;

template <typename T, bool L2>
__device__ __forceinline__ void chain_task(const DStep &st, int sub, int lane, const char *cbase, char *abase) {
  const T *Ap = region_ptr<T>(st.A, cbase, abase);
  const T *Bp = region_ptr<T>(st.B, cbase, abase);
  T *Cp = const_cast<T *>(region_ptr<T>(st.C, cbase, abase));
  const int split = st.split;
  const int64_t item = (int64_t)sub * 32 + lane;
  const int64_t c = item >> split;
  const int part = (int)(item & ((1 << split) - 1));
  const bool active = c < (int64_t(1) << st.nC);
  const T sum = warp_parts(active ? direct_part<T, L2>(st, (uint32_t)c, part, Ap, Bp) : czero<T>(), split);
  if (active && part == 0) Cp[c] = sum;
}

template <typename T>
__global__ void __launch_bounds__(kChainThreads) direct_chain_kernel(const DStep *steps, int n_steps, const int2 *tab,
                                                                     int n_levels, const char *cbase, char *abase) {
  __shared__ __align__(16) DStep s_st[kChainSteps];
  __shared__ int2 s_lv[kChainLevels];
  uint32_t rank, ctas;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(ctas));
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int w = (int)rank * kChainWarps + warp;
  // every level's bounds and every step's descriptor, read at once (fetched
  // level by level, each level waited for three dependent loads: 2.1 us a
  // level); a warp's task of the next level is read before the barrier
  for (int i = threadIdx.x; i < n_steps * (int)(sizeof(DStep) / 16); i += kChainThreads)
    reinterpret_cast<uint4 *>(s_st)[i] = reinterpret_cast<const uint4 *>(steps)[i];
  for (int i = threadIdx.x; i < n_levels; i += kChainThreads) s_lv[i] = tab[i];
  const int2 *tasks = tab + n_levels;
  __syncthreads();
  int2 lv = s_lv[0], task = w < lv.y ? tasks[lv.x + w] : make_int2(0, 0);
  for (int l = 0; l < n_levels; l++) {
    const int2 next = l + 1 < n_levels ? s_lv[l + 1] : make_int2(0, 0);
    const int2 ntask = w < next.y ? tasks[next.x + w] : make_int2(0, 0);
    if (w < lv.y) {
      if (ctas == 1)
        chain_task<T, false>(s_st[task.x], task.y, lane, cbase, abase);
      else
        chain_task<T, true>(s_st[task.x], task.y, lane, cbase, abase);
    }
    if (l + 1 == n_levels) break;
    lv = next;
    task = ntask;
    if (ctas == 1)
      __syncthreads();
    else
      asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}

int chain_tasks(const DStep &st) { return std::max(1, (1 << (st.nC + st.split)) / 32); }

int chain_ctas(int max_tasks) {
  int c = 1;
  while (c < 8 && c * kChainWarps < max_tasks) c *= 2;
  return c;
}

cudaError_t launch_direct_chain(const DStep *steps, int n_steps, const int *tab, int n_levels, int ctas,
                                const char *cbase, char *abase, int dbl, cudaStream_t s) {
  if (n_steps > kChainSteps || n_levels > kChainLevels || ctas * kChainWarps > kChainTasks) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)ctas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)ctas);
  cfg.blockDim = dim3(kChainThreads);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const int2 *t2 = reinterpret_cast<const int2 *>(tab);
  const cudaError_t e = dbl ? cudaLaunchKernelEx(&cfg, direct_chain_kernel<double2>, steps, n_steps, t2, n_levels, cbase,
                                              abase)
                            : cudaLaunchKernelEx(&cfg, direct_chain_kernel<float2>, steps, n_steps, t2, n_levels, cbase,
                                              abase);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// ---------------------------------------------------------------- queue
// The persistent form. ctrl[0] hands out tickets (the launch's blocks in
// order), ctrl[1] counts blocks that have left, ctrl[2] is the stop flag,
// ctrl[3] is a counter nothing increments (the test stall waits on it), and
// ctrl[4 + j] counts the finished blocks of step j.
//
// Progress: a step's blocks come after the blocks of the steps it reads
// (DStep::dep < own index, tickets in block order). A block holding a
// ticket is resident, so the lowest unfinished ticket always has all of its
// inputs done and runs to the end; no wait can close a cycle, whatever the
// grid size. Every wait is still bounded. Block b's first ticket is b itself
// (no atomic); later tickets come from ctrl[0], which starts at the grid size.
//
// Visibility: a producer block's threads write their results, meet at a
// barrier, and one thread fences and counts the block done; a consumer's
// waiting thread reads the count with acquire semantics at GPU scope before
// its block's barrier, so the block's plain loads that follow see the
// results (the acquire also keeps the SM's L1 from serving older copies).
// Results of one launch never share a 128-byte line with anything else read
// in it: the tensors of a queue launch all live through the whole launch, so
// none reuses another's memory, and every tensor starts on 256 bytes.
constexpr unsigned long long kQueueWaitNs = 2000000000ull;  // 2 s (default)
__device__ unsigned long long g_dq_wait_ns = kQueueWaitNs;
__device__ int g_dq_stall;

__device__ __forceinline__ unsigned long long dq_globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Wait until *cnt >= target: 1 when it is, 0 when the launch was stopped or
// the wait ran out (then the error word and the stop flag are set).
__device__ __forceinline__ bool dq_wait(const unsigned *cnt, unsigned target, unsigned *stop, int *err,
                                        unsigned long long limit) {
  if (ld_acquire(cnt) >= target) return true;
  const unsigned long long t0 = dq_globaltimer();
  for (unsigned polls = 1;; polls++) {
    if (ld_acquire(cnt) >= target) return true;
    if ((polls & 15) == 0) {
      if (ld_acquire(stop)) return false;
      if (dq_globaltimer() - t0 > limit) {
        atomicExch(err, 1);
        atomicExch(stop, 1u);
        return false;
      }
      if (polls >= 256) __nanosleep(32);
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(256) direct_queue_kernel(const DStep *steps, int n_steps, const int *bmap,
                                                           int64_t total, const char *cbase, char *abase,
                                                           unsigned *ctrl, int *err) {
  __shared__ int s_idx, s_go, s_last;
  __shared__ int64_t s_blk;
  __shared__ __align__(16) DStep s_st;
  __shared__ T red[256];
  unsigned *done = ctrl + 4;
  const unsigned long long limit = g_dq_wait_ns;
  // thread 0 takes the block's next ticket as soon as it has passed the
  // waits of the current one, so the atomic's latency hides behind the
  // block's work (a block holds at most one ticket it has not started, and
  // every ticket below it is finished or running: progress is unchanged)
  int64_t t_next = blockIdx.x;
  for (;;) {
    if (threadIdx.x == 0) {
      const int64_t t = t_next;
      int go = t < total;
      int idx = 0;
      if (go) {
        idx = bmap[t];
        if (g_dq_stall && t == 0) go = dq_wait(&ctrl[3], 1u, &ctrl[2], err, limit);
        const int4 dp = *reinterpret_cast<const int4 *>(steps[idx].dep);  // dep[2], dep_nblk[2]
        if (go && dp.x >= 0) go = dq_wait(&done[dp.x], (unsigned)dp.z, &ctrl[2], err, limit);
        if (go && dp.y >= 0) go = dq_wait(&done[dp.y], (unsigned)dp.w, &ctrl[2], err, limit);
        if (go) t_next = (int64_t)gridDim.x + atomicAdd(&ctrl[0], 1u);
      }
      s_idx = idx;
      s_blk = t;
      s_go = go;
    }
    __syncthreads();
    if (!s_go) break;
    stage_step(&s_st, steps + s_idx);
    __syncthreads();
    direct_block<T>(s_st, s_blk - s_st.block_begin, cbase, abase, red);
    __syncthreads();  // every result of this block is written
    if (threadIdx.x == 0) {
      __threadfence();
      atomicAdd(&done[s_idx], 1u);
    }
  }
  // the last block to leave zeroes the counters for the next launch
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(&ctrl[1], 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (s_last) {
    __threadfence();
    for (int j = threadIdx.x; j < n_steps; j += blockDim.x) done[j] = 0;
    __syncthreads();
    if (threadIdx.x == 0) {
      ctrl[0] = 0;
      ctrl[2] = 0;
      ctrl[3] = 0;
      __threadfence();
      ctrl[1] = 0;
    }
  }
}

namespace {
// resident blocks of the queue kernel per device (blocks per SM x SMs)
std::mutex g_dq_mu;
int g_dq_resident[2][64];
}  // namespace

template <typename T>
static int dq_resident(int dbl) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  std::lock_guard<std::mutex> lk(g_dq_mu);
  int &r = g_dq_resident[dbl][dev];
  if (r == 0) {
    int per_sm = 0, sms = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, direct_queue_kernel<T>, 256, 0) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      return 0;
    r = std::max(1, per_sm) * std::max(1, sms);
  }
  return r;
}

cudaError_t launch_direct_queue(const DStep *steps, int n_steps, const int *bmap, int64_t total_blocks,
                                const char *cbase, char *abase, unsigned *ctrl, int *err, int dbl, cudaStream_t s) {
  if (n_steps <= 0) return cudaSuccess;
  if (total_blocks > 0x7fffffffLL || !ctrl || !err || !bmap) return cudaErrorInvalidValue;
  const int resident = dbl ? dq_resident<double2>(1) : dq_resident<float2>(0);
  if (resident <= 0) return cudaErrorInvalidDevice;
  const unsigned grid = (unsigned)std::min<int64_t>(total_blocks, resident);
  if (dbl)
    direct_queue_kernel<double2><<<grid, 256, 0, s>>>(steps, n_steps, bmap, total_blocks, cbase, abase, ctrl, err);
  else
    direct_queue_kernel<float2><<<grid, 256, 0, s>>>(steps, n_steps, bmap, total_blocks, cbase, abase, ctrl, err);
  return cudaGetLastError();
}

cudaError_t direct_queue_set_wait_limit(unsigned long long ns) {
  const unsigned long long v = ns ? ns : kQueueWaitNs;
  return cudaMemcpyToSymbol(g_dq_wait_ns, &v, sizeof(v));
}

cudaError_t direct_queue_set_stall(int on) {
  const int v = on ? 1 : 0;
  return cudaMemcpyToSymbol(g_dq_stall, &v, sizeof(v));
}

// acc[row][o] += scale * root[beta, o] in FP64 for the current chunk (o the
// value of the open output qubits; m = 0 without them); then advance the
// group state (next slice, wrapping to the next chunk).
template <typename T>
__global__ void accum_kernel(AccumArgs a) {
  const T *root = static_cast<const T *>(a.root);
  GroupState *gs = a.gs;
  // everything the state says, in one round of loads
  const int64_t chunk = gs->chunk, n_rows = gs->n_rows, slice = gs->slice, lo = gs->lo, hi = gs->hi,
                done = gs->groups_done;
  const int tc_error = gs->tc_error;
  const int total = 1 << (a.g + a.m);
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const int beta = e >> a.m, o = e & ((1 << a.m) - 1);
    int64_t off = 0;
    for (int j = 0; j < a.g; j++) off |= int64_t((beta >> j) & 1) << a.beta_pos[j];
    for (int j = 0; j < a.m; j++) off |= int64_t((o >> j) & 1) << a.open_pos[j];
    const int64_t row = (chunk << a.g) | beta;
    if (row < n_rows) {
      const T v = root[off];
      const double vr = v.x, vi = v.y;
      const int64_t at = (row << a.m) | o;
      double2 r = a.acc[at];
      r.x += a.scale_re * vr - a.scale_im * vi;
      r.y += a.scale_re * vi + a.scale_im * vr;
      // a product of this call timed out: its rows are poisoned, so a
      // caller that only reads the amplitudes still sees the failure
      if (tc_error) r = make_double2(__longlong_as_double(0x7ff8000000000000ll),
                                         __longlong_as_double(0x7ff8000000000000ll));
      a.acc[at] = r;
    }
  }
  if (gridDim.x > 1) return;  // the state advances in a launch of its own
  __syncthreads();
  if (threadIdx.x == 0 && a.advance) {
    int64_t sl = slice + 1;
    if (sl >= hi) {
      sl = lo;
      gs->chunk = chunk + 1;
    }
    gs->slice = sl;
    gs->groups_done = done + 1;
  }
}

__global__ void advance_kernel(GroupState *gs) {
  int64_t sl = gs->slice + 1;
  if (sl >= gs->hi) {
    sl = gs->lo;
    gs->chunk = gs->chunk + 1;
  }
  gs->slice = sl;
  gs->groups_done++;
}

// one block up to 4096 root values; beyond, one value per thread over
// several blocks, and a separate launch advances the state once they are done
constexpr int kAccumOneBlock = 12;

int accumulate_launches(int g, int m) { return g + m <= kAccumOneBlock ? 1 : 2; }

cudaError_t launch_accumulate(const AccumArgs &a, cudaStream_t s) {
  if (a.g < 0 || a.m < 0 || a.g > kMaxBatch || a.m > kMaxOpen) return cudaErrorInvalidValue;
  const int bits = a.g + a.m;
  const unsigned blocks = bits <= kAccumOneBlock ? 1u : (unsigned)(((1 << bits) + 255) / 256);
  if (a.dbl)
    accum_kernel<double2><<<blocks, 256, 0, s>>>(a);
  else
    accum_kernel<float2><<<blocks, 256, 0, s>>>(a);
  if (blocks > 1 && a.advance) advance_kernel<<<1, 1, 0, s>>>(a.gs);
  return cudaGetLastError();
}

__global__ void accum_plain_kernel(const float2 *part, double2 *acc, int64_t n, double sre, double sim) {
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
    const double vr = part[j].x, vi = part[j].y;
    double2 r = acc[j];
    r.x += sre * vr - sim * vi;
    r.y += sre * vi + sim * vr;
    acc[j] = r;
  }
}

cudaError_t launch_accumulate_plain(const float2 *part, double2 *acc, int64_t n, double sre, double sim,
                                    cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  int64_t blocks = (n + 255) / 256;
  if (blocks > 65536) blocks = 65536;
  accum_plain_kernel<<<(unsigned)blocks, 256, 0, s>>>(part, acc, n, sre, sim);
  return cudaGetLastError();
}

}  // namespace dev
}  // namespace tz
