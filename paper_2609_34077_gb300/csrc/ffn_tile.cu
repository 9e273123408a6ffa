// Expert FFN of fp32 layers whose segments hold several rows: CUDA-core fp32 GEMM tiles.
//
// F(x) = W2 (silu(W1 x) * (W3 x)) per expert segment (Section 3.1; SwiGLU experts), in fp32 throughout.
// The row-streaming kernels (ffn_rowwise.cu) read each weight row once per 8 tokens and load 16 bytes
// of activations per four multiply-adds and token, which suits segments of a few tokens; beyond that
// those loads bound them. Here a CTA of 128 threads computes 64 tokens x 32 outputs (GEMM13: 32 gate
// and the 32 up values of the same outputs, joined in registers): 32 contraction elements per step,
// copied to shared memory three steps ahead (cp.async, rows padded by 16 bytes), 4 tokens x 8 (GEMM13)
// or 4 (GEMM2) values per thread, so 12 (8) 16-byte shared loads feed 128 (64) multiply-adds.
// 8 products are summed first, 4 such sums make a step's, and what adding a step to the total drops is
// carried into the next step (compensated summation): one running sum's error grows with the square root
// of its length, and the row-wise kernels add 32 lanes' short sums in a tree. Error of a dot product of
// normal values against 64 bits: 7.4e-8 at every length, row-wise 8.1e-8 at 256 and 1.2e-7 at 1024
// elements (8.8e-8 and 1.3e-7 with the steps simply added, 6 % faster).
// Measured (GB300, d = 256, w = 512, 8 experts, 512 tokens on 4 of them, events around each launch):
// GEMM13 35 us and GEMM2 29 us against 168 and 179 us row-wise; the multiply-adds alone take 11 us at
// the fp32 rate: the tile counts (256 and 128) leave the SMs few warps to hide shared loads behind.
// Warps take 16 tokens each, and one without tokens skips its arithmetic.
#include "common.cuh"
#include "internal.h"

namespace mcft {
namespace {

constexpr int kThreads = 128;
constexpr int TM = 64;   // tokens per tile
constexpr int BK = 32;   // contraction elements per step
constexpr int TN = 32;   // outputs per tile
constexpr int kDepth = 4;       // steps in shared memory, three of them on their way
constexpr int kPitch = BK + 4;  // floats per shared row

struct Items {
  int total;
  int off[kMaxSeg + 1];
  int first[kMaxSeg + 1];  // first item of each segment
};

// Work list: every non-empty segment of this launch's phase in ceil(rows / 64) x (outputs / 32) items
// (three segments per lane of the calling warp).
__device__ void build_items(Items& it, const FfnArgs& a, int outs) {
  const int lane = threadIdx.x & 31;
  const int nseg = a.hdr->abort == 0 ? a.nseg : 0;
  const unsigned long long hits = a.ready ? *a.ready : 0ull;
  for (int s = lane; s <= nseg; s += 32) it.off[s] = a.off[s];
  __syncwarp();
  int cnt[3], sum = 0;
  bool bad = false;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int s = lane * 3 + j;
    cnt[j] = 0;
    if (s < nseg) {
      const int n = it.off[s + 1] - it.off[s];
      if (n > 0 && seg_in_phase(a, s, hits)) {
        if (seg_block(a, s) == nullptr) bad = true;  // a selected expert without weights
        else cnt[j] = (n + TM - 1) / TM * (outs / TN);
      }
    }
    sum += cnt[j];
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
    const int s = lane * 3 + j;
    if (s <= nseg) it.first[s] = excl;
    excl += cnt[j];
  }
  const bool any_bad = __any_sync(0xffffffffu, bad);
  if (lane == 31) {
    if (any_bad) {
      set_error(a.err, kErrInvalid);
      const_cast<WsHeader*>(a.hdr)->abort = 1;
    }
    it.total = incl;
  }
}

__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}

// STAGE 13: h[q, j] = silu(W1[j] . x_t) * (W3[j] . x_t); STAGE 2: o[q, j] = W2[j] . h_q.
template <int STAGE>
constexpr int kNB = STAGE == 13 ? 2 * TN : TN;  // weight rows of a tile
template <int STAGE>
constexpr int kSmemBytes = kDepth * (TM + kNB<STAGE>) * kPitch * 4;

template <int STAGE>
__global__ void __launch_bounds__(kThreads, 3) ffn_tile_kernel(const __grid_constant__ FfnArgs a) {
  constexpr int NB = kNB<STAGE>, NC = NB / 8;  // weight rows per tile and per thread
  constexpr int LA = TM * BK / 4 / kThreads, LB = NB * BK / 4 / kThreads;  // 16-byte copies per thread
  constexpr int kStep = (TM + NB) * kPitch;
  __shared__ Items it;
  extern __shared__ __align__(16) float smem[];  // kDepth steps of [TM + NB rows][kPitch]
  pdl_wait();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int outs = STAGE == 13 ? a.w : a.d, K = STAGE == 13 ? a.d : a.w;
  if (warp == 0) build_items(it, a, outs);
  __syncthreads();
  const int kq = tid & 7, lr = tid >> 3;  // this thread's 16-byte column and first row of a copy
  // thread's tokens t0 + 4 i and weight rows c0 + 8 j: a quarter warp's 16-byte loads hit 32 banks
  const int t0 = warp * 16 + (lane >> 3), c0 = lane & 7;
  const int nseg = a.nseg, steps = K / BK;
  for (int item = blockIdx.x; item < it.total; item += gridDim.x) {
    int s = 0, hi = nseg - 1;  // the last segment whose first item is <= item: it has items
    while (s < hi) {
      const int mid = (s + hi + 1) >> 1;
      if (it.first[mid] <= item) s = mid;
      else hi = mid - 1;
    }
    const int rows = it.off[s + 1] - it.off[s], nt = (rows + TM - 1) / TM;
    const int local = item - it.first[s];
    const int r0 = local / nt * TN;                 // first output; token tiles innermost
    const int q0 = it.off[s] + local % nt * TM;     // first permuted row
    const int n = min(TM, it.off[s + 1] - q0);
    const float* blk = reinterpret_cast<const float*>(seg_block(a, s));
    const float* pa[LA];
    const float* pb[LB];
#pragma unroll
    for (int i = 0; i < LA; ++i) {  // rows past the end repeat the tile's first row and are dropped
      const int r = lr + i * (kThreads / 8), q = q0 + (r < n ? r : 0);
      pa[i] = STAGE == 13 ? reinterpret_cast<const float*>(a.x) + size_t(a.perm[q]) * K
                          : reinterpret_cast<const float*>(a.h) + size_t(q) * K;
      pa[i] += kq * 4;
    }
#pragma unroll
    for (int i = 0; i < LB; ++i) {
      const int r = lr + i * (kThreads / 8);
      const size_t row = STAGE == 13 ? size_t(r < TN ? r0 + r : a.w + r0 + r - TN) : size_t(r0 + r);
      pb[i] = blk + (STAGE == 13 ? size_t(0) : size_t(2) * a.w * a.d) + row * K + kq * 4;
    }
    auto copy = [&](int step) {  // one commit group per step, empty past the end
      if (step < steps) {
        float* d = smem + (step % kDepth) * kStep + lr * kPitch + kq * 4;
#pragma unroll
        for (int i = 0; i < LA; ++i) cp_async16(d + i * (kThreads / 8) * kPitch, pa[i] + step * BK);
#pragma unroll
        for (int i = 0; i < LB; ++i)
          cp_async16(d + (TM + i * (kThreads / 8)) * kPitch, pb[i] + step * BK);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float acc[4][NC], sum[4][NC];  // [token][weight row]: total, and the step's with what it lost
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < NC; ++j) acc[i][j] = sum[i][j] = 0.f;
    const bool busy = warp * 16 < n;
    __syncthreads();  // the previous item's steps are read
    for (int st = 0; st < kDepth - 1; ++st) copy(st);
    for (int st = 0; st < steps; ++st) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kDepth - 2) : "memory");
      __syncthreads();  // step st is in shared memory; everyone is done with step st - 1
      copy(st + kDepth - 1);
      if (busy) {
        const float* xa = smem + (st % kDepth) * kStep + t0 * kPitch;
        const float* wb = smem + (st % kDepth) * kStep + (TM + c0) * kPitch;
#pragma unroll
        for (int k8 = 0; k8 < BK; k8 += 8) {
          float part[4][NC];
#pragma unroll
          for (int k = k8; k < k8 + 8; k += 4) {
            float4 xv[4], wv[NC];
#pragma unroll
            for (int i = 0; i < 4; ++i) xv[i] = *reinterpret_cast<const float4*>(xa + 4 * i * kPitch + k);
#pragma unroll
            for (int j = 0; j < NC; ++j) wv[j] = *reinterpret_cast<const float4*>(wb + 8 * j * kPitch + k);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int j = 0; j < NC; ++j) {
                float p = k == k8 ? xv[i].x * wv[j].x : fmaf(xv[i].x, wv[j].x, part[i][j]);
                p = fmaf(xv[i].y, wv[j].y, p);
                p = fmaf(xv[i].z, wv[j].z, p);
                part[i][j] = fmaf(xv[i].w, wv[j].w, p);
              }
          }
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < NC; ++j) sum[i][j] += part[i][j];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < NC; ++j) {
            // what the addition drops stays in sum, for the next step (nothing beside an infinite total)
            const float t = acc[i][j] + sum[i][j], lost = sum[i][j] - (t - acc[i][j]);
            sum[i][j] = fabsf(t) < INFINITY ? lost : 0.f;
            acc[i][j] = t;
          }
      }
    }
    const void* lblk = a.lrank ? a.lblk[s] : nullptr;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (t0 + 4 * i >= n) continue;
      const int q = q0 + t0 + 4 * i;
      float* out = STAGE == 13 ? reinterpret_cast<float*>(a.h) + size_t(q) * a.w
                               : a.o + size_t(q) * a.d;
#pragma unroll
      for (int j = 0; j < TN / 8; ++j) {
        const int row = r0 + c0 + 8 * j;
        float g = acc[i][j] + sum[i][j];
        if constexpr (STAGE == 13) {
          float u = acc[i][j + TN / 8] + sum[i][j + TN / 8];
          if (lblk) {  // LoRA: + s B1 (A1 x), + s B3 (A3 x)
            const LoraOffsets lo = lora_offsets(a.d, a.w, a.lrank);
            const float* m = a.u13 + size_t(q) * 2 * a.lrank;
            g += lora_up<float>(lblk, lo.b1, row, m, a.lrank, a.lscale);
            u += lora_up<float>(lblk, lo.b3, row, m + a.lrank, a.lrank, a.lscale);
          }
          out[row] = silu(g) * u;
        } else {
          if (lblk)  // LoRA: + s B2 (A2 h)
            g += lora_up<float>(lblk, lora_offsets(a.d, a.w, a.lrank).b2, row,
                                a.u2 + size_t(q) * a.lrank, a.lrank, a.lscale);
          out[row] = g;
        }
      }
    }
  }
}

template <int STAGE>
cudaError_t launch_stage(const FfnArgs& a, int num_sms, cudaStream_t s) {
  static SmemOptIn smem;
  cudaError_t e = smem.allow(reinterpret_cast<const void*>(ffn_tile_kernel<STAGE>), kSmemBytes<STAGE>);
  if (e != cudaSuccess) return e;
  const int kid = STAGE == 13 ? kProfFfn13 : kProfFfn2;
  prof_begin(kid, s);
  e = launch_pdl(ffn_tile_kernel<STAGE>, dim3(3 * num_sms), dim3(kThreads), kSmemBytes<STAGE>, s, a);
  prof_end(kid, s);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

cudaError_t launch_ffn_tile(const FfnArgs& a, int num_sms, cudaStream_t s, int stages) {
  cudaError_t e = cudaSuccess;
  if (stages & 1) e = launch_stage<13>(a, num_sms, s);
  if (e != cudaSuccess || !(stages & 2)) return e;
  return launch_stage<2>(a, num_sms, s);
}

}  // namespace mcft
