// LoRA down-projections for the Stage-2 expert forward (Section 3.2: the experts are fine-tuned
// with LoRA adapters; rank 8 and alpha 16 in Appendix B).
//
// Each adapted projection is W v + s B (A v) with A [r, in], B [out, r], s = alpha / r. The large
// term W v runs in the expert GEMM / GEMV kernels, which also add s B u in their epilogues (r
// multiply-adds per output). On the decode and fp32 paths lora_down_kernel computes the small middle
// vectors u = A v for every permuted row whose segment has an adapter (the tensor-core path has
// lora_down_tile_kernel below, and adds B u as further k-blocks of its GEMMs):
//   stage 13: u[q] = [A1 x ; A3 x]     (2r values; x = the row's token, or the gathered row)
//   stage 2:  u[q] = A2 h_q            (r values; h = the SwiGLU activation of the row)
// One warp per row: lanes walk the input in 16-byte chunks, each chunk is dotted with the R rows
// of A (small, L1/L2-resident), and R warp reductions finish the row. Rows of segments without an
// adapter, and padding rows, get zeros.
#include "common.cuh"
#include "internal.h"

namespace mcft {
namespace {

constexpr int kWarps = 8;

template <typename T>
struct In16;  // 16 bytes of an input or adapter row as fp32
template <>
struct In16<__nv_bfloat16> {
  static constexpr int n = 8;
  __device__ static void load(const void* p, float* f) { unpack8(ldg16(p), f); }
};
template <>
struct In16<float> {
  static constexpr int n = 4;
  __device__ static void load(const void* p, float* f) {
    const uint4 v = ldg16(p);
    f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y);
    f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
  }
};

// T: dtype of the input rows and of the adapter (the layer dtype); R: outputs per row (2r or r).
template <typename T, int R>
__global__ void __launch_bounds__(kWarps * 32) lora_down_kernel(const __grid_constant__ LoraDownArgs a) {
  pdl_wait();
  __shared__ int s_off[kMaxSeg + 1];
  __shared__ int s_nseg;
  if (threadIdx.x == 0) s_nseg = a.hdr->abort == 0 ? a.nseg : 0;
  __syncthreads();
  const int nseg = s_nseg;
  for (int s = threadIdx.x; s <= nseg; s += blockDim.x) s_off[s] = a.off[s];
  __syncthreads();
  if (nseg == 0) return;
  const int mrows = s_off[nseg];
  const int lane = threadIdx.x & 31;
  using C = In16<T>;
  for (int q = blockIdx.x * kWarps + (threadIdx.x >> 5); q < mrows; q += gridDim.x * kWarps) {
    int s = 0;
    while (s + 1 < nseg && s_off[s + 1] <= q) ++s;
    const char* blk = reinterpret_cast<const char*>(a.lblk[s]);
    const int tok = a.row_tok[q];  // -1 for a padding row
    float* out = a.u + size_t(q) * a.ustride;
    if (blk == nullptr || tok < 0) {
      for (int j = lane; j < R; j += 32) out[j] = 0.f;
      continue;
    }
    const int src = a.by_token ? tok : q;  // x is indexed by token, h by permuted row
    const char* in = reinterpret_cast<const char*>(a.in) + size_t(src) * a.in_stride * sizeof(T);
    float acc[R];
#pragma unroll
    for (int j = 0; j < R; ++j) acc[j] = 0.f;
    for (int k = lane * C::n; k < a.K; k += 32 * C::n) {
      float xv[C::n];
      C::load(in + size_t(k) * sizeof(T), xv);
#pragma unroll
      for (int j = 0; j < R; ++j) {
        // adapter row j: rows of the first A (A1 or A2), then of the second (A3) at stage 13
        const size_t aoff = j < a.r ? a.a_off0 + size_t(j) * a.K : a.a_off1 + size_t(j - a.r) * a.K;
        float wv[C::n];
        C::load(blk + (aoff + k) * sizeof(T), wv);
#pragma unroll
        for (int i = 0; i < C::n; ++i) acc[j] = fmaf(wv[i], xv[i], acc[j]);
      }
    }
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const float v = warp_sum(acc[j]);
      if (lane == 0) out[j] = v;
    }
  }
}

// The down projections of the tensor-core path: U = s (A v) in bf16 for the rows of every segment
// with an adapter, [rows, NT * 8] ([s A1 x | s A3 x] or s A2 h), or with split = 3 [rows, 3 * NT * 8]: bf16
// of the fp32 values, of what that leaves of them, and of what is left then, which together hold all 24 bits.
// A skinny GEMM bound by
// reading v once: as in the router's tiles, a CTA takes 16 rows of one segment and its 8 warps one
// contraction slice each (mma.sync m16n8k16, U 32-element chunks of every operand in flight per
// lane), so 2000 rows are 125 CTAs; partial sums are added in shared memory in slice order.
constexpr int kTileRows = 16;
template <int NT, int U>
__global__ void __launch_bounds__(kWarps * 32, 2)
    lora_down_tile_kernel(const __grid_constant__ LoraDownArgs a) {
  pdl_wait();
  __shared__ int s_off[kMaxSeg + 1], s_first[kMaxSeg + 1];
  __shared__ float part[kWarps][kTileRows][NT * 8 + 1];
  if (a.hdr->abort) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
  const int nseg = a.nseg;
  if (warp == 0) {  // segment offsets and first tiles (three segments per lane)
    for (int s = lane; s <= nseg; s += 32) s_off[s] = a.off[s];
    __syncwarp();
    int cnt[3], sum = 0;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int s = lane * 3 + j;
      cnt[j] = s < nseg && a.lblk[s] ? (s_off[s + 1] - s_off[s] + kTileRows - 1) / kTileRows : 0;
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
      if (s <= nseg) s_first[s] = excl;
      excl += cnt[j];
    }
  }
  __syncthreads();
  const int nch = a.K / 32;
  const int c0 = warp * nch / kWarps, c1 = (warp + 1) * nch / kWarps;
  for (int tile = blockIdx.x; tile < s_first[nseg]; tile += gridDim.x) {
    int lo = 0, hi = nseg - 1;  // the last segment whose first tile is <= tile: it is not empty
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (s_first[mid] <= tile) lo = mid;
      else hi = mid - 1;
    }
    const int q0 = s_off[lo] + (tile - s_first[lo]) * kTileRows;
    const int n = min(kTileRows, s_off[lo + 1] - q0);
    const char* blk = reinterpret_cast<const char*>(a.lblk[lo]);
    // rows past the segment's end repeat its first row of the tile; their results are dropped
    auto src = [&](int r) -> const char* {
      const int q = q0 + (r < n ? r : 0);
      const int row = a.by_token ? max(a.row_tok[q], 0) : q;
      return reinterpret_cast<const char*>(a.in) + size_t(row) * a.in_stride * 2 + c * 16;
    };
    const char* xa = src(g);
    const char* xb = src(g + 8);
    const char* wr[NT];
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      const int o = j * 8 + g;  // output: a row of the first A (A1 or A2), then of the second (A3)
      wr[j] = blk + (o < a.r ? a.a_off0 + size_t(o) * a.K : a.a_off1 + size_t(o - a.r) * a.K) * 2 + c * 16;
    }
    float acc[NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
    for (int ch = c0; ch < c1; ch += U) {
      uint4 va[U], vb[U], vw[U][NT];
#pragma unroll
      for (int i = 0; i < U; ++i)
        if (ch + i < c1) {
          const size_t o = size_t(ch + i) * 64;
          va[i] = ldg16(xa + o);
          vb[i] = ldg16(xb + o);
#pragma unroll
          for (int j = 0; j < NT; ++j) vw[i][j] = ldg16(wr[j] + o);
        }
#pragma unroll
      for (int i = 0; i < U; ++i)
        if (ch + i < c1)
#pragma unroll
          for (int j = 0; j < NT; ++j) {
            mma16816(acc[j], va[i].x, vb[i].x, va[i].y, vb[i].y, vw[i][j].x, vw[i][j].y);
            mma16816(acc[j], va[i].z, vb[i].z, va[i].w, vb[i].w, vw[i][j].z, vw[i][j].w);
          }
    }
    __syncthreads();  // the previous tile's partial sums are read
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      const int o = j * 8 + 2 * c;
      part[warp][g][o] = acc[j][0];
      part[warp][g][o + 1] = acc[j][1];
      part[warp][g + 8][o] = acc[j][2];
      part[warp][g + 8][o + 1] = acc[j][3];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n * NT * 8; i += kWarps * 32) {
      const int r = i / (NT * 8), o = i % (NT * 8);
      float v = part[0][r][o];
#pragma unroll
      for (int k = 1; k < kWarps; ++k) v += part[k][r][o];
      v *= a.scale;
      uint16_t* u = reinterpret_cast<uint16_t*>(a.u) + size_t(q0 + r) * (a.split * NT * 8) + o;
      const bool finite = fabsf(v) < INFINITY;
      for (int i = 0; i < a.split; ++i) {
        uint16_t h = f2bf(v);
        if (finite && a.split > 1 && (h & 0x7fff) == 0x7f80) h -= 1;  // rounded past the largest number
        u[i * NT * 8] = h;
        v = finite ? v - bf16lo(h) : 0.f;
      }
    }
  }
}

template <typename T>
cudaError_t launch_typed(const LoraDownArgs& a, int outs, int blocks, cudaStream_t s) {
  switch (outs) {
    case 8: lora_down_kernel<T, 8><<<blocks, kWarps * 32, 0, s>>>(a); break;
    case 16: lora_down_kernel<T, 16><<<blocks, kWarps * 32, 0, s>>>(a); break;
    case 32: lora_down_kernel<T, 32><<<blocks, kWarps * 32, 0, s>>>(a); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_lora_down_tiles(const LoraDownArgs& a, int outs, int mcap, int num_sms, cudaStream_t s) {
  const int cap = (mcap + kTileRows - 1) / kTileRows + a.nseg;  // most tiles there can be
  const dim3 grid(cap < 4 * num_sms ? cap : 4 * num_sms), block(kWarps * 32);
  prof_begin(kProfLora, s);
  const cudaError_t e = outs == 8    ? launch_pdl(lora_down_tile_kernel<1, 6>, grid, block, 0, s, a)
                        : outs == 16 ? launch_pdl(lora_down_tile_kernel<2, 4>, grid, block, 0, s, a)
                        : outs == 32 ? launch_pdl(lora_down_tile_kernel<4, 3>, grid, block, 0, s, a)
                                     : cudaErrorInvalidValue;
  prof_end(kProfLora, s);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_lora_down(const LoraDownArgs& a, int dtype, int outs, int mcap, cudaStream_t s) {
  int blocks = (mcap + kWarps - 1) / kWarps;
  if (blocks > 4096) blocks = 4096;
  if (blocks < 1) blocks = 1;
  prof_begin(kProfLora, s);
  const cudaError_t e = dtype == MCFT_BF16 ? launch_typed<__nv_bfloat16>(a, outs, blocks, s)
                                           : launch_typed<float>(a, outs, blocks, s);
  prof_end(kProfLora, s);
  return e;
}

}  // namespace mcft
