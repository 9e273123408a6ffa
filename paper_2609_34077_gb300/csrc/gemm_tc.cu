// Grouped expert GEMMs with the tokens on the MMA's M side, on CTA pairs (tcgen05 + TMEM, fed by TMA):
// the tile shape that mcft_set_tc_tiles(MCFT_TC_TILES_CTA_PAIR) selects. The default is gemm_rows.cu.
//
// Section 3.1: each routed expert is F(x) = W2 (silu(W1 x) * (W3 x)) (SwiGLU); with tokens
// permuted into per-expert segments (padded to 256 rows), the two expert GEMMs of a layer are
//   GEMM13: acc[m, 0:128] = xp[m] . W1[n0:n0+128]^T, acc[m, 128:256] = xp[m] . W3[n0:n0+128]^T,
//           h[m, n0:n0+128] = bf16(silu(acc_gate) * acc_up)             (fused epilogue)
//   GEMM2:  o[m, n0:n0+256] = h[m] . W2[n0:n0+256]^T                       (fp32 out)
// both D = A B^T with A and B K-major bf16, fp32 accumulators in tensor memory.
//
// Tiles of 256 rows x 256 columns, one MMA of M = 256 per K step issued by the pair's leader over both
// CTAs' shared memory. Each CTA loads its 128 activation rows and its half of the tile's 256 weight
// rows (GEMM13: rank 0 the W1 rows, rank 1 the W3 rows, i.e. the gate and up halves of N; GEMM2: 128
// consecutive W2 rows each), so every weight element is read from shared memory once for the rows of
// both CTAs. 6 stages of 32 KB:
//   warp 0 (both CTAs) - TMA producer (one thread); the loads of both CTAs complete on the leader's
//             full[s], on which the leader expects the pair's bytes; each CTA waits on its own empty[s];
//   warp 1 - allocates the pair's TMEM (both CTAs), two 128 x 256 fp32 accumulators each; in the
//             leader, issues the MMAs, whose commits arrive on empty[s] and tfull[b] of both CTAs;
//   warps 2-5 (both CTAs) - epilogue of the CTA's 128 rows of the tile: tcgen05.ld of their 32-lane
//             quarter, SwiGLU or fp32, staged through shared memory and stored as whole 128-byte row
//             segments; they release the accumulator on the leader's tempty[b] (eight arrivals: four
//             warps per CTA), so the next tile's MMAs overlap this tile's epilogue.
// Tiles are walked m-fastest inside groups of m-tiles so concurrently running pairs share weight
// tiles (and the activation group) in L2. Every wait is bounded: after 2 s the kernel records
// MCFT_ERR_TIMEOUT, stops issuing, waits (bounded) for its copies and MMAs in flight, frees TMEM
// and returns. The leader drains its last stages' copies (both CTAs' bytes), the peer waits (bounded)
// until its last stages were consumed, and both CTAs leave through one cluster barrier after the
// leader's MMAs have completed, so neither exits while the other may still read its shared memory or
// arrive on its barriers.
#include <cuda.h>

#include "common.cuh"
#include "internal.h"
#include "mbar.cuh"
#include "tc_ptx.cuh"

namespace mcft {
namespace {

constexpr int BM = 128, BN = 256, BK = 64;
constexpr int A_BYTES = BM * BK * 2;
constexpr int kPairRows = 2 * BM;
constexpr int kPairStages = 6;
constexpr int kPairStageBytes = A_BYTES + (BN / 2) * BK * 2;  // 128 activation + 128 weight rows
constexpr int kPairTmemCols = 2 * BN;                          // two 128 x 256 accumulators
// Instruction descriptor, kind::f16: D fp32 (bits 4-5 = 1), A bf16 (bits 7-9 = 1), B bf16
// (bits 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 at bit 17, M >> 4 at bit 24.
constexpr uint32_t kPairIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(BN >> 3) << 17) |
                                (uint32_t(kPairRows >> 4) << 24);
constexpr int kThreads = 192;  // producer, MMA, 4 epilogue warps

enum { EPI_SWIGLU = 0, EPI_F32 = 1 };

struct TcParams {
  CUtensorMap tma_a;
  CUtensorMap tma_b[kMaxSeg];
  const int* off;
  const WsHeader* hdr;
  void* out;
  unsigned* err;
  uint32_t wmask[3];  // segments that have weights
  int nseg, kblocks, ntiles_n, ldo, b_half, group_m;
};

struct SmemCtl {
  uint64_t full[kPairStages], empty[kPairStages], tfull[2], tempty[2], drain;
  uint32_t tmem_base;
  int abort;
  int mt_total;
  int nseg;
  int off[kMaxSeg + 1];
};

// Epilogue store staging: each epilogue warp writes 32 rows x 128 bytes of its
// output into shared memory (rows padded to 144 bytes: conflict-free 16-byte writes and reads),
// then stores them as whole 128-byte row segments, four rows per instruction.
constexpr int kOutRowBytes = 144;
constexpr int kOutWarpBytes = 32 * kOutRowBytes;
constexpr int kCtlBytes = (int(sizeof(SmemCtl)) + 15) / 16 * 16;
constexpr int kPairSmem = kPairStages * kPairStageBytes + 1024 + kCtlBytes + 4 * kOutWarpBytes;
static_assert(kPairSmem <= 227 * 1024, "shared memory");

// Tile -> (m-tile, n-tile): groups of group_m m-tiles; inside a group, n-major then m.
__device__ __forceinline__ void tile_coords(int tile, int mt_total, int ntn, int G, int& mt,
                                            int& nt) {
  const int g = tile / (G * ntn);
  const int r = tile - g * G * ntn;
  const int gsz = min(G, mt_total - g * G);
  nt = r / gsz;
  mt = g * G + r % gsz;
}

__device__ __forceinline__ int seg_of_row(const SmemCtl* c, int row) {
  int s = 0;
  while (s + 1 < c->nseg && c->off[s + 1] <= row) ++s;
  return s;
}

// Epilogue of one expert-GEMM tile for the 32 accumulator rows of an epilogue warp (TMEM lane
// quarter at taddr, output rows grow0 .. grow0 + 31, n-tile nt): SwiGLU to bf16 h (GEMM13) or fp32
// (GEMM2), staged through the warp's shared rows stg and stored as whole 128-byte row segments.
template <int EPI, int NB>
__device__ __forceinline__ void store_tile(const TcParams& p, uint8_t* stg, uint32_t taddr,
                                           size_t grow0, int nt, int lane) {
  if constexpr (EPI == EPI_SWIGLU) {
    // two rounds of 64 h columns (128 bytes of bf16 per row)
#pragma unroll 1
    for (int c0 = 0; c0 < NB / 2; c0 += 64) {
#pragma unroll
      for (int c = 0; c < 64; c += 16) {
        uint32_t g[16], u[16];
        tmem_ld16(taddr + c0 + c, g);
        tmem_ld16(taddr + NB / 2 + c0 + c, u);
        tmem_ld_wait();
        uint32_t pk[8];
        bool regular = true;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          regular &= silu_regular(__uint_as_float(g[2 * i])) && silu_regular(__uint_as_float(g[2 * i + 1]));
          pk[i] = pack2bf(silu_branchless(__uint_as_float(g[2 * i])) * __uint_as_float(u[2 * i]),
                          silu_branchless(__uint_as_float(g[2 * i + 1])) * __uint_as_float(u[2 * i + 1]));
        }
        if (!regular) {  // rare: this lane's values again, by IEEE division
#pragma unroll
          for (int i = 0; i < 8; ++i)
            pk[i] = pack2bf(silu(__uint_as_float(g[2 * i])) * __uint_as_float(u[2 * i]),
                            silu(__uint_as_float(g[2 * i + 1])) * __uint_as_float(u[2 * i + 1]));
        }
        uint4* sw = reinterpret_cast<uint4*>(stg + lane * kOutRowBytes + c * 2);
        sw[0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
        sw[1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
      }
      __syncwarp();
      const size_t col = size_t(nt) * (NB / 2) + c0 + (lane & 7) * 8;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int r = 4 * i + (lane >> 3);
        const uint4 v = *reinterpret_cast<const uint4*>(stg + r * kOutRowBytes + (lane & 7) * 16);
        *reinterpret_cast<uint4*>(reinterpret_cast<uint16_t*>(p.out) + (grow0 + r) * p.ldo + col) = v;
      }
      __syncwarp();
    }
  } else {
    // eight rounds of 32 fp32 columns (128 bytes per row)
#pragma unroll 1
    for (int c0 = 0; c0 < NB; c0 += 32) {
#pragma unroll
      for (int c = 0; c < 32; c += 16) {
        uint32_t v[16];
        tmem_ld16(taddr + c0 + c, v);
        tmem_ld_wait();
        uint4* sw = reinterpret_cast<uint4*>(stg + lane * kOutRowBytes + c * 4);
#pragma unroll
        for (int i = 0; i < 4; ++i) sw[i] = make_uint4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
      }
      __syncwarp();
      const size_t col = size_t(nt) * NB + c0 + (lane & 7) * 4;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int r = 4 * i + (lane >> 3);
        const uint4 v = *reinterpret_cast<const uint4*>(stg + r * kOutRowBytes + (lane & 7) * 16);
        *reinterpret_cast<uint4*>(reinterpret_cast<float*>(p.out) + (grow0 + r) * p.ldo + col) = v;
      }
      __syncwarp();
    }
  }
}

template <int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    gemm_tc_pair_kernel(const __grid_constant__ TcParams p) {
  pdl_wait();
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;  // the same offsets in both CTAs
  SmemCtl* ctl =
      reinterpret_cast<SmemCtl*>(smem_raw + (base - raw) + kPairStages * kPairStageBytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const bool leader = rank == 0;

  if (threadIdx.x == 0) {
    // both CTAs find the same offsets and the same abort decision
    int abort = p.hdr->abort;
    const int nseg = p.nseg;
    ctl->nseg = nseg;
    for (int s = 0; s <= nseg; ++s) ctl->off[s] = p.off[s];
    for (int s = 0; s < nseg; ++s) {
      if (ctl->off[s + 1] > ctl->off[s] && !((p.wmask[s >> 5] >> (s & 31)) & 1u)) {
        set_error(p.err, kErrInvalid);  // a selected expert without weights
        const_cast<WsHeader*>(p.hdr)->abort = 1;
        abort = 1;
      }
    }
    ctl->abort = abort;
    ctl->mt_total = abort ? 0 : ctl->off[nseg] / kPairRows;
    for (int s = 0; s < kPairStages; ++s) {
      mbar_init(&ctl->full[s], 1);
      mbar_init(&ctl->empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&ctl->tfull[b], 1);
      mbar_init(&ctl->tempty[b], 8);
    }
    mbar_init(&ctl->drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&ctl->tmem_base)),
                 "r"(kPairTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  cluster_sync();  // barriers initialised and TMEM allocated in both CTAs
  tc_fence_after();

  const uint32_t tmem = ctl->tmem_base;
  const int mt_total = ctl->mt_total;  // 256-row tiles
  const int ntn = p.ntiles_n;
  const int tiles = mt_total * ntn;
  const int cid = int(blockIdx.x >> 1), ncl = int(gridDim.x >> 1);  // pair, pairs
  volatile int* abort = &ctl->abort;

  if (warp == 0) {
    if (cid < tiles && elect_one()) {
      uint32_t it = 0;
      for (int tile = cid; tile < tiles && !*abort; tile += ncl) {
        int mt, nt;
        tile_coords(tile, mt_total, ntn, p.group_m, mt, nt);
        const CUtensorMap* mb = &p.tma_b[seg_of_row(ctl, mt * kPairRows)];
        const int row0 = mt * kPairRows + int(rank) * BM;
        const int yb = EPI == EPI_SWIGLU ? int(rank) * p.b_half + nt * (BN / 2)
                                         : nt * BN + int(rank) * (BN / 2);
        for (int kb = 0; kb < p.kblocks; ++kb, ++it) {
          const int s = int(it % kPairStages);
          if (!mbar_wait_cl(&ctl->empty[s], ((it / kPairStages) & 1u) ^ 1u, abort, p.err)) break;
          const uint32_t sa = base + uint32_t(s) * kPairStageBytes, sb = sa + A_BYTES;
          const uint32_t fb = peer_addr(&ctl->full[s], 0);
          if (leader) mbar_expect_tx(&ctl->full[s], 2 * kPairStageBytes);
          tma_load_2d_pair(sa, &p.tma_a, kb * BK, row0, fb);
          tma_load_2d_pair(sb, mb, kb * BK, yb, fb);
        }
      }
      // Stages still in flight: the leader waits for their bytes (both CTAs'), the peer until
      // the leader's MMAs consumed them; after the first wait that runs out (an aborted pair,
      // 2 s: nothing is in flight any more) the rest are skipped.
      const uint32_t n_tail = it < kPairStages ? it : kPairStages;
      for (uint32_t j = it - n_tail; j < it; ++j) {
        uint64_t* bar = leader ? &ctl->full[j % kPairStages] : &ctl->empty[j % kPairStages];
        if (!mbar_wait_drain_cl(bar, (j / kPairStages) & 1u, p.err)) break;
      }
    }
  } else if (warp == 1) {
    if (leader && cid < tiles && elect_one()) {
      uint32_t it = 0, lt = 0;
      for (int tile = cid; tile < tiles && !*abort; tile += ncl) {
        const uint32_t b = lt & 1u;
        if (!mbar_wait_cl(&ctl->tempty[b], ((lt >> 1) & 1u) ^ 1u, abort, p.err)) break;
        tc_fence_after();
        const uint32_t dt = tmem + b * BN;
        bool ok = true;
        for (int kb = 0; kb < p.kblocks; ++kb, ++it) {
          const int s = int(it % kPairStages);
          if (!mbar_wait_cl(&ctl->full[s], (it / kPairStages) & 1u, abort, p.err)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sa = base + uint32_t(s) * kPairStageBytes, sb = sa + A_BYTES;
          const uint64_t da = sw128_desc(sa), db = sw128_desc(sb);
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)
            tc_mma_pair(dt, da + uint64_t(2 * k), db + uint64_t(2 * k), kPairIdesc,
                        (kb | k) != 0 ? 1u : 0u);
          tc_commit_pair_both(&ctl->empty[s]);
        }
        if (!ok) break;
        tc_commit_pair_both(&ctl->tfull[b]);
        ++lt;
      }
      tc_commit_pair(&ctl->drain);  // arrives once every MMA issued above has completed
      mbar_wait_drain_cl(&ctl->drain, 0, p.err);
    }
  } else if (warp >= 2 && warp < 6) {
    const int q = warp & 3;  // TMEM lane quarter this warp may access
    uint8_t* stg = reinterpret_cast<uint8_t*>(ctl) + kCtlBytes + q * kOutWarpBytes;
    uint32_t lt = 0;
    for (int tile = cid; tile < tiles; tile += ncl) {
      int mt, nt;
      tile_coords(tile, mt_total, ntn, p.group_m, mt, nt);
      const uint32_t b = lt & 1u;
      int ok = 1;
      if (lane == 0) ok = mbar_wait_cl(&ctl->tfull[b], (lt >> 1) & 1u, abort, p.err) ? 1 : 0;
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) break;
      tc_fence_after();
      const uint32_t taddr = tmem + b * BN + (uint32_t(q * 32) << 16);
      const size_t grow0 = size_t(mt) * kPairRows + rank * BM + q * 32;
      store_tile<EPI, BN>(p, stg, taddr, grow0, nt, lane);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(peer_addr(&ctl->tempty[b], 0));
      ++lt;
    }
  }

  tc_fence_before();
  cluster_sync();  // the leader's MMAs drained, every copy landed, both epilogues done
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(kPairTmemCols)
                 : "memory");
  }
}

// bf16 matrix [rows, cols] row-major; box 64 columns (128 B, one swizzle span) x 128 rows.
bool encode_2d(CUtensorMap* m, const void* base, uint64_t cols, uint64_t rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn || (reinterpret_cast<uintptr_t>(base) & 15u) || ((cols * 2) & 15u)) return false;
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {cols * 2};
  const cuuint32_t box[2] = {BK, 128};
  const cuuint32_t es[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// With CTA-pair tiles selected, layers whose routed experts average at least this many rows run
// on pairs (segments padded to 256 rows); with fewer the extra padding would dominate.
constexpr int kPairMinRows = 512;

int group_for(size_t a_tile_bytes, size_t budget_mb) {
  const size_t budget = budget_mb << 20;  // activation rows kept hot in L2 per group
  size_t g = budget / (a_tile_bytes ? a_tile_bytes : 1);
  return g < 1 ? 1 : int(g > 4096 ? 4096 : g);
}

// One pair per two SMs that can hold one at a time (one CTA per SM): a persistent grid of pairs
// that all run at once, so no pair's tiles wait for another pair to exit.
template <int EPI>
cudaError_t launch_pair(const TcParams& p, int num_sms, cudaStream_t s) {
  static SmemOptIn smem;
  static ResidentClusters resident;
  const void* fn = reinterpret_cast<const void*>(gemm_tc_pair_kernel<EPI>);
  const cudaError_t e = smem.allow(fn, kPairSmem);
  if (e != cudaSuccess) return e;
  const int pairs = resident.get(fn, num_sms & ~1, kThreads, kPairSmem);
  if (pairs < 1) return cudaErrorInvalidConfiguration;
  const int kid = EPI == EPI_SWIGLU ? kProfGemm13Pair : kProfGemm2Pair;
  prof_begin(kid, s);
  gemm_tc_pair_kernel<EPI><<<2 * pairs, kThreads, kPairSmem, s>>>(p);
  prof_end(kid, s);
  return cudaGetLastError();
}

}  // namespace

bool tc_pair_tiles(int T, int K, int E, int lrank) {
  return lrank == 0 && size_t(T) * K >= size_t(kPairMinRows) * E;
}

cudaError_t launch_ffn_tc(const FfnArgs& a, const void* xp, int mcap, int pad, int num_sms,
                          cudaStream_t s, int stages) {
  if (pad != kPairRows || a.lrank != 0) return cudaErrorInvalidValue;
  TcParams p13, p2;
  memset(&p13, 0, sizeof(p13));
  memset(&p2, 0, sizeof(p2));
  const size_t d = size_t(a.d), w = size_t(a.w);
  if (!encode_2d(&p13.tma_a, xp, d, size_t(mcap))) return cudaErrorInvalidValue;
  if (!encode_2d(&p2.tma_a, a.h, w, size_t(mcap))) return cudaErrorInvalidValue;
  for (int sgi = 0; sgi < a.nseg; ++sgi) {
    const char* blk = reinterpret_cast<const char*>(a.wblk[sgi]);
    if (!blk) continue;
    if (!encode_2d(&p13.tma_b[sgi], blk, d, 2 * w)) return cudaErrorInvalidValue;
    if (!encode_2d(&p2.tma_b[sgi], blk + 2 * w * d * 2, w, d)) return cudaErrorInvalidValue;
    p13.wmask[sgi >> 5] |= 1u << (sgi & 31);
  }
  p2.wmask[0] = p13.wmask[0];
  p2.wmask[1] = p13.wmask[1];
  p2.wmask[2] = p13.wmask[2];
  for (TcParams* q : {&p13, &p2}) {
    q->off = a.off;
    q->hdr = a.hdr;
    q->err = a.err;
    q->nseg = a.nseg;
  }
  p13.out = a.h;
  p13.kblocks = int(d / BK);
  p13.ntiles_n = int(w / (BN / 2));
  p13.ldo = int(w);
  p13.b_half = int(w);
  // L2 budgets per group of m-tiles, from sweeps over the Mixtral-shaped T = 4096 layer
  p13.group_m = group_for(size_t(pad) * d * 2, 24);
  p2.out = a.o;
  p2.kblocks = int(w / BK);
  p2.ntiles_n = int(d / BN);
  p2.ldo = int(d);
  p2.b_half = 0;
  p2.group_m = group_for(size_t(pad) * w * 2, 12);
  cudaError_t e = cudaSuccess;
  if (stages & 1) e = launch_pair<EPI_SWIGLU>(p13, num_sms, s);
  if (e != cudaSuccess || !(stages & 2)) return e;
  return launch_pair<EPI_F32>(p2, num_sms, s);
}

}  // namespace mcft
