// Token permutation by expert: histogram, exclusive scan of padded segment sizes, and a stable
// scatter (assignments keep their (t, k) order inside each expert), plus the spread of the activations
// into the permuted matrix for the tensor-core path. Segments E..E+S-1 hold the shared
// experts, which process every token (Section 3.1). The stable order defines the result uniquely,
// so the one-CTA kernel (decode and other small batches) and the cluster write the same rows.
#include <cooperative_groups.h>

#include "common.cuh"
#include "internal.h"

namespace cg = cooperative_groups;

namespace mcft {
namespace {

constexpr int kThreads = 1024;

// Padded exclusive scan of the segment sizes by warp 0 (three segments per lane, kMaxSeg <= 96):
// writes offs (shared) and, if asked, a.off, a.cnt and the header.
__device__ void scan_segments(const PermuteArgs& a, const int* hist, int* offs, int lane,
                              bool write = true) {
  const int nseg = a.E + a.S;
  int len[3], padded[3], sum = 0;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int sg = lane * 3 + j;
    len[j] = sg < nseg ? (sg < a.E ? hist[sg] : a.T) : 0;
    padded[j] = (len[j] + a.pad - 1) / a.pad * a.pad;
    sum += padded[j];
  }
  int incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  int excl = incl - sum;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int sg = lane * 3 + j;
    if (sg < nseg) {
      offs[sg] = excl;
      if (write) {
        a.off[sg] = excl;
        a.cnt[sg] = len[j];
      }
    }
    excl += padded[j];
  }
  if (lane == 31) {
    offs[nseg] = incl;
    if (write) {
      a.off[nseg] = incl;
      a.hdr->abort = 0;
      a.hdr->nseg = nseg;
      a.hdr->mrows = incl;
    }
  }
}

// Stable scatter of assignments [i0, i1) (all threads of the CTA, kThreads of them): each
// assignment's row is offs[e] + run[e] + (earlier assignments of e in this round); run[e] holds the
// number of earlier assignments of e before the round and is advanced by it.
__device__ void scatter_rounds(const PermuteArgs& a, int i0, int i1, const int* offs, int* run,
                               int (*wcnt)[kMaxE]) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  for (int base = i0; base < i1; base += kThreads) {
    const int i = base + tid;
    const bool valid = i < i1;
    const int e = valid ? a.idx[i] : -1;
    for (int j = tid; j < (kThreads / 32) * kMaxE; j += kThreads) (&wcnt[0][0])[j] = 0;
    __syncthreads();
    const unsigned peers = __match_any_sync(0xffffffffu, e);
    const int rank = __popc(peers & lt_mask);
    if (valid && rank == 0) wcnt[warp][e] = __popc(peers);
    __syncthreads();
    if (valid) {
      int p = run[e] + rank;
      for (int w = 0; w < warp; ++w) p += wcnt[w][e];
      const int row = offs[e] + p;
      a.pos[i] = row;
      a.perm[row] = i / a.K;
    }
    __syncthreads();
    if (tid < a.E) {
      int tot = 0;
      for (int w = 0; w < kThreads / 32; ++w) tot += wcnt[w][tid];
      run[tid] += tot;
    }
    __syncthreads();
  }
}

// Padding rows of routed segments (-1) and the rows of shared segments (every token in order):
// rows r0, r0 + stride, ... of [0, mrows); a row's segment is found by binary search on offs.
__device__ void fill_rows(const PermuteArgs& a, const int* offs, const int* len_of, int r0,
                          int stride) {
  const int nseg = a.E + a.S;
  const int mrows = offs[nseg];
  for (int r = r0; r < mrows; r += stride) {
    int lo = 0, hi = nseg;  // largest segment with offs[seg] <= r
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (offs[mid] <= r) lo = mid;
      else hi = mid;
    }
    const int len = lo < a.E ? len_of[lo] : a.T;
    const int local = r - offs[lo];
    if (lo >= a.E && local < len) a.perm[r] = local;
    else if (local >= len) a.perm[r] = -1;
  }
}

// One CTA for the whole call (decode batches, and up to 1024 assignments: a few microseconds).
__global__ void __launch_bounds__(kThreads) permute_kernel(const __grid_constant__ PermuteArgs a) {
  pdl_wait();
  // the next launch (the decode FFN) may start now: before its own wait it reads only what was
  // written before this kernel started (its parameters, the cache's expert table)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __shared__ int hist[kMaxSeg];
  __shared__ int run[kMaxE];
  __shared__ int offs[kMaxSeg + 1];
  __shared__ int wcnt[kThreads / 32][kMaxE];
  __shared__ int bad;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = a.T * a.K, nseg = a.E + a.S;
  if (tid < kMaxSeg) hist[tid] = 0;
  if (tid < kMaxE) run[tid] = 0;
  if (tid == 0) bad = 0;
  __syncthreads();
  for (int i = tid; i < n; i += kThreads) {
    const int e = a.idx[i];
    if (e < 0 || e >= a.E) bad = 1;
    else atomicAdd(&hist[e], 1);
  }
  __syncthreads();
  // progress and claim counters: on every path, the abort path included
  if (a.done && tid < nseg + kClaimSlots) a.done[tid] = 0;
  if (bad) {
    if (tid == 0) {
      a.hdr->abort = 1;
      a.hdr->mrows = 0;
      set_error(a.err, kErrInvalid);
    }
    return;
  }
  if (warp == 0) scan_segments(a, hist, offs, lane);
  __syncthreads();
  scatter_rounds(a, 0, n, offs, run, wcnt);
  fill_rows(a, offs, hist, tid, kThreads);
}

// Larger calls: the same permutation by one cluster of 8 CTAs. Each of its 256 warps takes a
// contiguous stretch of the assignments and counts them per expert (its own row of counters, so no
// atomics); the counters of a CTA's warps and then, over distributed shared memory, of the CTAs are
// scanned per expert; every CTA scans the segment sizes for itself; and each warp walks its stretch again
// and places it. A chain of dependent steps bounds it, not the 100 KB of ids. ncu, GB300: T = 4096 with
// K = 6 8.1 us against 15.4 for a count, a scan and a scatter launch (K = 2: 5.5 / 12), T = 16384 with K = 6
// 16.7 / 17.2, and 1200 assignments (T = 200) 6.2 us against 8.6 for the one-CTA kernel above, which walks
// 1024 assignments at a time. Up to one such walk that kernel is the faster one: whole forwards of small layers,
// cluster / one CTA: 65 assignments 16.9 / 16.0 us, 512 17.8 / 17.0, 1024 18.7 / 18.3, 1500 18.9 / 20.1 (64 experts).
// At decode sizes it stays too: it lets the FFN start beside it.
constexpr int kPermCtas = 8;
constexpr int kPermWarps = kThreads / 32;
constexpr int kPermAhead = 4;  // rounds of ids loaded together

// Lanes of the warp whose id (>= 0, below 2^bits) equals this lane's: one ballot per bit, several
// times the rate of match.any with tens of different ids in a warp.
__device__ __forceinline__ unsigned same_id(int id, int bits) {
  unsigned peers = __ballot_sync(0xffffffffu, id >= 0);
  for (int b = 0; b < bits; ++b) {
    const unsigned m = __ballot_sync(0xffffffffu, (id >> b) & 1);
    peers &= (id >> b) & 1 ? m : ~m;
  }
  return peers;
}

__global__ void __cluster_dims__(kPermCtas, 1, 1) __launch_bounds__(kThreads)
    permute_cluster_kernel(const __grid_constant__ PermuteArgs a) {
  __shared__ int wcnt[kPermWarps][kMaxE + 1];  // per warp: its counts, then its first position
  __shared__ int ctot[kMaxE];                  // this CTA's count per expert (read by the others)
  __shared__ int cbad;                         // this CTA saw an id out of range (read by the others)
  __shared__ int hist[kMaxSeg], base[kMaxE], offs[kMaxSeg + 1];
  __shared__ int bad;
  cg::cluster_group cluster = cg::this_cluster();
  const int crank = int(cluster.block_rank());
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  const int n = a.T * a.K, nseg = a.E + a.S, E = a.E;
  const int bits = 32 - __clz(E - 1);  // (E = 1: 0, every id is the same)
  for (int j = tid; j < kPermWarps * (kMaxE + 1); j += kThreads) (&wcnt[0][0])[j] = 0;
  if (tid == 0) cbad = bad = 0;
  pdl_wait();
  __syncthreads();
  // this warp's assignments [i0, i1), whole rounds of 32
  const int rounds = (n + kPermCtas * kThreads - 1) / (kPermCtas * kThreads);
  const int i0 = (crank * kPermWarps + warp) * rounds * 32, i1 = min(n, i0 + rounds * 32);
  for (int b = i0; b < i1; b += 32 * kPermAhead) {
    int id[kPermAhead];
#pragma unroll
    for (int j = 0; j < kPermAhead; ++j) {
      const int i = b + 32 * j + lane;
      id[j] = i < i1 ? a.idx[i] : -1;
      if (i < i1 && (id[j] < 0 || id[j] >= E)) {
        cbad = 1;
        id[j] = -1;
      }
    }
#pragma unroll
    for (int j = 0; j < kPermAhead; ++j) {
      if (b + 32 * j >= i1) break;
      const unsigned peers = same_id(id[j], bits);
      if (id[j] >= 0 && (peers & lt_mask) == 0) wcnt[warp][id[j]] += __popc(peers);
      __syncwarp();
    }
  }
  __syncthreads();
  for (int e = warp; e < E; e += kPermWarps) {  // lane = warp: exclusive scan over the CTA's warps
    const int c = wcnt[lane][e];
    int v = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += u;
    }
    wcnt[lane][e] = v - c;
    if (lane == 31) ctot[e] = v;
  }
  cluster.sync();  // every CTA's counts are in its shared memory
  if (tid < E) {
    int before = 0, all = 0;
#pragma unroll
    for (int r = 0; r < kPermCtas; ++r) {
      const int c = *cluster.map_shared_rank(&ctot[tid], r);
      before += r < crank ? c : 0;
      all += c;
    }
    base[tid] = before;
    hist[tid] = all;
  } else if (tid >= kMaxE && tid < kMaxE + kPermCtas) {
    if (*cluster.map_shared_rank(&cbad, tid - kMaxE)) bad = 1;
  }
  __syncthreads();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");  // done with the others' memory
  // progress and claim counters: on every path, the abort path included
  if (crank == 0 && a.done && tid < nseg + kClaimSlots) a.done[tid] = 0;
  if (bad) {
    if (crank == 0 && tid == 0) {
      a.hdr->abort = 1;
      a.hdr->mrows = 0;
      set_error(a.err, kErrInvalid);
    }
  } else {
    if (warp == 0) scan_segments(a, hist, offs, lane, crank == 0);
    __syncthreads();
    for (int b = i0; b < i1; b += 32 * kPermAhead) {
      int id[kPermAhead];
#pragma unroll
      for (int j = 0; j < kPermAhead; ++j) {
        const int i = b + 32 * j + lane;
        id[j] = i < i1 ? a.idx[i] : -1;
      }
#pragma unroll
      for (int j = 0; j < kPermAhead; ++j) {
        if (b + 32 * j >= i1) break;
        const int e = id[j];
        const unsigned peers = same_id(e, bits);
        const int rank = __popc(peers & lt_mask);
        const int p = e >= 0 ? wcnt[warp][e] : 0;
        __syncwarp();
        if (e >= 0) {
          if (rank == 0) wcnt[warp][e] = p + __popc(peers);
          const int i = b + 32 * j + lane, row = offs[e] + base[e] + p + rank;
          a.pos[i] = row;
          if (!a.spread) a.perm[row] = i / a.K;
        }
        __syncwarp();
      }
    }
    // rows of the shared experts (every token in order), and the padding rows (-1)
    const int ct = crank * kThreads + tid;
    for (int s = 0; s < a.S; ++s)
      for (int t = ct; t < a.T; t += kPermCtas * kThreads) a.perm[offs[E + s] + t] = t;
    if (a.pad > 1)
      for (int s = crank * kPermWarps + warp; s < nseg; s += kPermCtas * kPermWarps)
        for (int r = offs[s] + (s < E ? hist[s] : a.T) + lane; r < offs[s + 1]; r += 32) a.perm[r] = -1;
  }
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // nor the others with this CTA's
}

// The permuted activations of the tensor-core path: xp[pos[t, k], :] = x[t, :] (bf16), and
// perm[pos[t, k]] = t. One warp per token and 256 16-byte chunks of its row: the row is read once, eight
// loads in flight per lane, and written K times, which bounds it. With padded segments (gemm_tc.cu) also
// the shared experts' copies (off[E + s] + t) and zeros in the padding rows. Read by destination row, as
// this kernel's predecessor did, x comes from L2 K times, and the permutation has to scatter perm from
// its one cluster. ncu, GB300, DeepSeek-V2-Lite shape: T = 4096 29 -> 17.9 us (5.6 TB/s written),
// 16384 138 -> 71, 200 7.0 -> 3.8; Mixtral shape, T = 4096 14.9 -> 14.9.
constexpr int kSpreadWarps = 8;
__global__ void __launch_bounds__(kSpreadWarps * 32) spread_kernel(const __grid_constant__ SpreadArgs a) {
  pdl_wait();
  if (a.hdr->abort) return;
  const int nch = a.d / 8;  // 16-byte chunks per row
  const int parts = (nch + 255) / 256;
  const int lane = threadIdx.x & 31;
  const int w = blockIdx.x * kSpreadWarps + (threadIdx.x >> 5), nw = gridDim.x * kSpreadWarps;
  const int ncopy = a.K + (a.pad > 1 ? a.S : 0);  // (unpadded segments: the GEMM reads shared rows in x)
  uint4* xp = reinterpret_cast<uint4*>(a.xp);
  for (int i = w; i < a.T * parts * a.groups; i += nw) {
    const int t = i / (parts * a.groups), pg = i - t * (parts * a.groups);
    const int k0 = pg % a.groups, c0 = pg / a.groups * 256 + lane;
    int row = 0;
    if (lane < a.K) row = a.pos[size_t(t) * a.K + lane];
    else if (lane < ncopy) row = a.off[a.E + lane - a.K] + t;
    const uint4* src = reinterpret_cast<const uint4*>(a.x) + size_t(t) * nch;
    uint4 v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (c0 + 32 * j < nch) v[j] = ldg16(src + c0 + 32 * j);
    if (lane < a.K && c0 < 32 && k0 == 0) a.perm[row] = t;
    for (int k = k0; k < ncopy; k += a.groups) {
      uint4* dst = xp + size_t(__shfl_sync(0xffffffffu, row, k)) * nch;
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (c0 + 32 * j < nch) dst[c0 + 32 * j] = v[j];
    }
  }
  if (a.pad > 1)
    for (int s = 0; s < a.E + a.S; ++s)
      for (int r = a.off[s] + a.cnt[s] + w; r < a.off[s + 1]; r += nw)
        for (int c = lane; c < nch; c += 32) xp[size_t(r) * nch + c] = make_uint4(0, 0, 0, 0);
}

}  // namespace

cudaError_t launch_permute(const PermuteArgs& a, cudaStream_t s) {
  prof_begin(kProfPermute, s);
  cudaError_t e;
  if (a.T <= kPermDecodeT || a.T * a.K <= kThreads) {
    e = launch_pdl(permute_kernel, dim3(1), dim3(kThreads), 0, s, a);
  } else {
    e = launch_pdl(permute_cluster_kernel, dim3(kPermCtas), dim3(kThreads), 0, s, a);
  }
  prof_end(kProfPermute, s);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_spread(const SpreadArgs& args, cudaStream_t s) {
  SpreadArgs a = args;
  // a token's copies are shared out over warps while there are few tokens: 8 warps per SM or more
  const int tokens = a.T * ((a.d / 8 + 255) / 256);
  a.groups = max(1, min(a.K, 8 * num_sms() / tokens));
  const int items = tokens * a.groups;
  const int need = (items + kSpreadWarps - 1) / kSpreadWarps, most = 8 * num_sms();
  prof_begin(kProfGather, s);
  const cudaError_t e = launch_pdl(spread_kernel, dim3(need < most ? need : most),
                                   dim3(kSpreadWarps * 32), 0, s, a);
  prof_end(kProfGather, s);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace mcft
